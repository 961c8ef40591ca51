// broad.cu -- stage (a): broad phase at the full activation (Sec. 3.3).
//
// Canonical result: every non-incident primitive pair whose FP64 boxes, each
// inflated by h, overlap on all three axes (closed intervals).  The tests work
// on FP32 boxes rounded outward from the FP64 ones (lo rounded down, hi up), so
// FP32 overlap is implied by FP64 overlap: the FP32 pairs are a superset.  A
// pair is then accepted outright when the FP32 test still passes after moving
// every FP32 bound one ulp inward (the FP64 bound lies within that ulp),
// rejected when the plain FP32 test fails, and decided on the FP64 boxes
// (formed again from the positions) otherwise.
//
// The paper hashes primitives into cells.  Here the boxes are large beside the
// mesh (the activation spans several edges), so a cell hash holds every
// primitive about ten times, sorts those entries on every call and tests a
// pair in every cell it shares.  Instead each scene fixes an order of its
// primitives in which neighbours stay near each other however the mesh folds,
// and cuts it into clusters of 32 and
// superclusters of 32 clusters.  A call computes the boxes bottom up, pairs
// overlapping superclusters, then their clusters, and tests each pair of
// clusters (a tile) with one warp: lane = row primitive, a loop over the column
// primitives that reach the row cluster's box.  Each pair of primitives is
// tested in exactly one tile, nothing is sorted, and the tile writes its pairs
// where one atomicAdd per tile places them.  The only host wait is the read of
// the pair count.
//
// The order goes by component first, since the rest shape says nothing about
// where one component lies beside another (instances of one sheet share it, and
// are placed only through x).  Inside a component: triangles, edges and vertices
// along a Morton curve of the rest shape, yarn edges along their yarn.  A
// component that fills its clusters to three quarters has them to itself; the
// others (short fibres, confetti, single vertices) are packed behind each other
// along a Morton curve of their places, at rest to begin with.  Where those say
// nothing either, a call finds many more overlapping clusters than a scene in
// good order has, and packs them again by their places at its x (broad_phase).
// 20,000 fibres in random order, a pass: 66.5 -> 1.44 ms with 31 edges each, 15.2
// -> 0.63 with 8 (clusters across the fibres' ends in the caller's order before);
// 16 instances of a 40x40 sheet 2.65 -> 1.04 (one Morton curve over all of them
// before); 64 rod scenes 4.19 -> 3.97.
//
// Several scenes can share one pass (a batch): every member has its own box
// inflation, clusters never span members, and superclusters are paired within
// a member only, so primitives of different members never meet.
//
// Measured on GB300, contact_build (cell hash, sorted and swept in x -> tiles):
// pleated 256x256 sheet (14.8M candidates) 1.73 -> 0.24 ms, 200k-triangle graded
// disk (26.1M) 2.81 -> 0.49, 64 rod scenes (7.2M) 1.60 -> 0.32, woven patch of
// 4,112 vertices 0.17 -> 0.04 (some 30 launches and three host waits -> four
// and one).
#include <algorithm>
#include <cmath>
#include <numeric>
#include <vector>

#include "frest.cuh"
#include "prims.cuh"
#include "scene.cuh"

namespace {

__device__ __forceinline__ uint32_t f2o(float f) {
  uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float o2f(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

constexpr unsigned FULL = 0xffffffffu;
constexpr int CL = 32;  // primitives per cluster and clusters per supercluster: a warp's lanes

// the FP64 box of a primitive (vertex ids v, unused ones negative) at x, or
// over the sweep x -> x + p, before inflation
__device__ __forceinline__ void prim_box(const int4& v, int n, const double* __restrict__ x,
                                         const double* __restrict__ p, double (&lo)[3], double (&hi)[3]) {
  const int id[3] = {v.x, v.y, v.z};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double mn = INFINITY, mx = -INFINITY;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (id[a] < 0) continue;
      const double c = x[(size_t)k * n + id[a]];
      mn = fmin(mn, c);
      mx = fmax(mx, c);
      if (p) {
        const double c2 = xadd(c, p[(size_t)k * n + id[a]]);
        mn = fmin(mn, c2);
        mx = fmax(mx, c2);
      }
    }
    lo[k] = mn;
    hi[k] = mx;
  }
}

__device__ __forceinline__ double inflation(const MemberParams& m, bool swept) { return 0.5 * (swept ? m.xi : m.a); }

struct Box {
  float4 lo, hi;  // w unused
};
__device__ __forceinline__ Box load_box(const float4* __restrict__ b, int64_t i) { return Box{b[2 * i], b[2 * i + 1]}; }
__device__ __forceinline__ bool overlap(const Box& a, const Box& b) {
  return a.lo.x <= b.hi.x && b.lo.x <= a.hi.x && a.lo.y <= b.hi.y && b.lo.y <= a.hi.y && a.lo.z <= b.hi.z &&
         b.lo.z <= a.hi.z;
}
// the union of the lanes' boxes, in every lane
__device__ __forceinline__ void warp_union(Box& b) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    b.lo.x = fminf(b.lo.x, __shfl_xor_sync(FULL, b.lo.x, o));
    b.lo.y = fminf(b.lo.y, __shfl_xor_sync(FULL, b.lo.y, o));
    b.lo.z = fminf(b.lo.z, __shfl_xor_sync(FULL, b.lo.z, o));
    b.hi.x = fmaxf(b.hi.x, __shfl_xor_sync(FULL, b.hi.x, o));
    b.hi.y = fmaxf(b.hi.y, __shfl_xor_sync(FULL, b.hi.y, o));
    b.hi.z = fmaxf(b.hi.z, __shfl_xor_sync(FULL, b.hi.z, o));
  }
}
__device__ __forceinline__ Box empty_box() {
  return Box{make_float4(INFINITY, INFINITY, INFINITY, 0.f), make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f)};
}

// per member: [0..2] min (ordered), [3..5] max (ordered)
constexpr int BOUNDS_STRIDE = 6;

// One thread per vertex: its FP32 box (swept: of x and x + p inflated by xi / 2,
// the CCD phase; else of x inflated by a / 2, the full activation), each side
// the FP64 value rounded outwards.  Rounding and the inflation's sum keep the
// order of their operands, so the FP32 union of a primitive's vertex boxes is
// the primitive's FP64 box, inflated and rounded outwards, bit for bit -- with
// the FP64 work once per vertex instead of once per primitive and vertex of it
// (both broad phases of a pass: 200k-triangle graded sheet 108 -> 42 us, pleated
// 256x256 76 -> 35, 64 rod scenes 179 -> 106).
__global__ void __launch_bounds__(256) k_vertex_boxes(int n, bool swept, const double* __restrict__ x,
                                                      const double* __restrict__ p, const int32_t* __restrict__ vsc,
                                                      const MemberParams* __restrict__ mp, int members,
                                                      float4* __restrict__ lo, float4* __restrict__ hi) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double h = inflation(mp[members > 1 ? vsc[i] : 0], swept);
  float l[3], u[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double c = x[(size_t)k * n + i];
    double mn = c, mx = c;
    if (p) {
      const double q = p[(size_t)k * n + i], c2 = xadd(c, q);
      const bool back = __double_as_longlong(q) < 0;
      mn = back ? c2 : c;
      mx = back ? c : c2;
    }
    l[k] = __double2float_rd(xsub(mn, h));
    u[k] = __double2float_ru(xadd(mx, h));
    if (isnan(l[k]) || isnan(u[k])) {  // a NaN end takes no part
      mn = fmin((double)INFINITY, c);
      mx = fmax(-(double)INFINITY, c);
      if (p) {
        const double c2 = xadd(c, p[(size_t)k * n + i]);
        mn = fmin(mn, c2);
        mx = fmax(mx, c2);
      }
      l[k] = __double2float_rd(xsub(mn, h));
      u[k] = __double2float_ru(xadd(mx, h));
    }
  }
  lo[i] = make_float4(l[0], l[1], l[2], 0.f);
  hi[i] = make_float4(u[0], u[1], u[2], 0.f);
}

// A warp per cluster: the boxes of its primitives and their union.  box_raw
// (per-stencil activation) gets the uninflated FP64 boxes, by primitive.  Block
// 0 resets what the next kernels accumulate into.
struct BoxArgs {
  int nc, n, T, members;
  bool rod, swept;
  const int4* __restrict__ slots;
  const uint32_t* __restrict__ cinfo;  // member << 2 | group
  const double* __restrict__ x;
  const double* __restrict__ p;
  const MemberParams* __restrict__ mp;
  const float4* __restrict__ vlo;      // the vertices' boxes (null: from x and p)
  const float4* __restrict__ vhi;
  float4* __restrict__ box;
  float4* __restrict__ cbox;
  double* __restrict__ box_raw;
  uint32_t* __restrict__ bounds;
  unsigned long long* __restrict__ sc;      // scalars, those of the bits in `clear` set to 0
  uint32_t clear;
};

__global__ void __launch_bounds__(256) k_boxes(BoxArgs A) {
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i < A.members * BOUNDS_STRIDE; i += blockDim.x)
      A.bounds[i] = i % BOUNDS_STRIDE < 3 ? 0xffffffffu : 0u;
    if (threadIdx.x < SC_N && ((A.clear >> threadIdx.x) & 1u)) A.sc[threadIdx.x] = 0ull;
  }
  const int c = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (c >= A.nc) return;
  const int64_t s = (int64_t)c * CL + lane;
  const int4 v = A.slots[s];
  const uint32_t ci = A.cinfo[c];
  Box b = empty_box();
  if (v.w >= 0) {
    double lo[3], hi[3];
    if (A.box_raw || !A.vlo) prim_box(v, A.n, A.x, A.p, lo, hi);
    if (A.box_raw) {
      // broad-phase primitive ids: vertices, then triangles, then edges (rods: edges)
      const uint32_t g = ci & 3u;
      const int64_t q = A.rod || g == 0u ? v.w : (g == 1u ? (int64_t)A.n + v.w : (int64_t)A.n + A.T + v.w);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        A.box_raw[q * 6 + k] = lo[k];
        A.box_raw[q * 6 + 3 + k] = hi[k];
      }
    }
    if (!A.vlo) {
      const double h = inflation(A.mp[ci >> 2], A.swept);
      b.lo = make_float4(__double2float_rd(xsub(lo[0], h)), __double2float_rd(xsub(lo[1], h)),
                         __double2float_rd(xsub(lo[2], h)), 0.f);
      b.hi = make_float4(__double2float_ru(xadd(hi[0], h)), __double2float_ru(xadd(hi[1], h)),
                         __double2float_ru(xadd(hi[2], h)), 0.f);
    } else {
      const int id[3] = {v.x, v.y, v.z};
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (id[a] < 0) continue;
        const float4 l = A.vlo[id[a]], u = A.vhi[id[a]];
        b.lo = make_float4(fminf(b.lo.x, l.x), fminf(b.lo.y, l.y), fminf(b.lo.z, l.z), 0.f);
        b.hi = make_float4(fmaxf(b.hi.x, u.x), fmaxf(b.hi.y, u.y), fmaxf(b.hi.z, u.z), 0.f);
      }
    }
  }
  A.box[2 * s] = b.lo;
  A.box[2 * s + 1] = b.hi;
  warp_union(b);
  if (lane == 0) {
    A.cbox[2 * (int64_t)c] = b.lo;
    A.cbox[2 * (int64_t)c + 1] = b.hi;
  }
}

// A warp per supercluster: the union of its clusters' boxes, added to its
// member's bounds.  sup: first cluster, count, member.
__global__ void __launch_bounds__(256) k_super_boxes(int ns, const int4* __restrict__ sup,
                                                     const float4* __restrict__ cbox, float4* __restrict__ sbox,
                                                     uint32_t* __restrict__ bounds) {
  const int s = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (s >= ns) return;
  const int4 S = sup[s];
  Box b = lane < S.y ? load_box(cbox, (int64_t)S.x + lane) : empty_box();
  warp_union(b);
  if (lane == 0) {
    sbox[2 * (int64_t)s] = b.lo;
    sbox[2 * (int64_t)s + 1] = b.hi;
    uint32_t* q = bounds + (size_t)S.z * BOUNDS_STRIDE;
    atomicMin(&q[0], f2o(b.lo.x));
    atomicMin(&q[1], f2o(b.lo.y));
    atomicMin(&q[2], f2o(b.lo.z));
    atomicMax(&q[3], f2o(b.hi.x));
    atomicMax(&q[4], f2o(b.hi.y));
    atomicMax(&q[5], f2o(b.hi.z));
  }
}

// A block per job (a row supercluster against up to 32 column ones): the pairs
// of overlapping clusters, appended to tiles (counted past the capacity, not
// written).  The warps take the overlapping columns in turn: few jobs have any,
// those near the diagonal have most of theirs, and one warp per job left the
// chip waiting for the fullest (both broad phases of a pass: 200k-triangle
// graded sheet 202 -> 70 us, pleated 256x256 74 -> 34, 64 rod scenes 213 -> 57).
// Block 0 also forms each member's box centre and half its largest extent (cx;
// the origin of the FP32 positions).
constexpr int PAIR_WARPS = 8;
__global__ void __launch_bounds__(32 * PAIR_WARPS) k_cluster_pairs(int nj, const int4* __restrict__ jobs,
                                                       const int4* __restrict__ sup, const float4* __restrict__ sbox,
                                                       const float4* __restrict__ cbox, uint2* __restrict__ tiles,
                                                       unsigned long long cap, unsigned long long* __restrict__ ntiles,
                                                       int members, const uint32_t* __restrict__ bounds,
                                                       double* __restrict__ cx) {
  if (blockIdx.x == 0)
    for (int m = threadIdx.x; m < members; m += blockDim.x) {
      double X = 0.0, ctr[3];
      bool none = false;
      for (int k = 0; k < 3; ++k) {
        const double lo = o2f(bounds[m * BOUNDS_STRIDE + k]), hi = o2f(bounds[m * BOUNDS_STRIDE + 3 + k]);
        none |= !(hi >= lo);
        ctr[k] = 0.5 * (lo + hi);
        X = fmax(X, 0.5 * (hi - lo) * (1.0 + 1e-6));
      }
      for (int k = 0; k < 3; ++k) cx[4 * m + k] = none ? 0.0 : ctr[k];
      cx[4 * m + 3] = none ? 0.0 : X;
    }
  __shared__ Box rows[CL];
  const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5;
  for (int j = blockIdx.x; j < nj; j += gridDim.x) {
    const int4 J = jobs[j];  // row, first column, end of columns
    const int4 R = sup[J.x];
    __syncthreads();  // the last job's reads are over
    if (wb == 0) rows[lane] = lane < R.y ? load_box(cbox, (int64_t)R.x + lane) : empty_box();
    const Box rb = load_box(sbox, J.x);
    unsigned todo = __ballot_sync(FULL, J.y + lane < J.z && overlap(rb, load_box(sbox, min(J.y + lane, J.z - 1))));
    __syncthreads();
    for (int turn = 0; todo; ++turn) {
      const int col = J.y + __ffs((int)todo) - 1;
      todo &= todo - 1u;
      if ((turn & (PAIR_WARPS - 1)) != wb) continue;  // the block's warps take the columns in turn
      const int4 C = sup[col];
      const Box cb = lane < C.y ? load_box(cbox, (int64_t)C.x + lane) : empty_box();
      unsigned mine = 0u;  // the columns of row `lane`
#pragma unroll 8
      for (int r = 0; r < CL; ++r) {
        unsigned m = __ballot_sync(FULL, lane < C.y && overlap(rows[r], cb));
        if (J.x == col) m &= FULL << r;  // each pair of clusters once (and the cluster with itself)
        if (lane == r && r < R.y) mine = m;  // (an empty box's bounds do meet an infinite box's: the counts decide)
      }
      const unsigned cnt = (unsigned)__popc(mine);
      unsigned inc = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += u;
      }
      const unsigned total = __shfl_sync(FULL, inc, 31);
      if (total == 0) continue;
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(ntiles, (unsigned long long)total);
      base = __shfl_sync(FULL, base, 0) + inc - cnt;
      for (; mine; mine &= mine - 1u, ++base)
        if (base < cap) tiles[base] = make_uint2((uint32_t)(R.x + lane), (uint32_t)(C.x + __ffs((int)mine) - 1));
    }
  }
}

struct TileArgs {
  int n;
  bool rod, swept, canonical;
  int bi, bj;                        // compact keys: bits of the two indices
  const int4* __restrict__ slots;
  const uint32_t* __restrict__ cinfo;
  const float4* __restrict__ box;
  const float4* __restrict__ cbox;
  const uint2* __restrict__ tiles;
  const unsigned long long* __restrict__ ntiles;
  unsigned long long tile_cap;
  const double* __restrict__ x;
  const double* __restrict__ p;
  const MemberParams* __restrict__ mp;
  uint64_t* __restrict__ out;
  unsigned long long out_cap;
  unsigned long long* __restrict__ total;
  unsigned long long* fpstat;        // [0] FP32-accepted pairs, [1] FP64-decided (may be null)
  unsigned int* novf;                // rods: rows with more than half of a cluster as partners
  uint8_t* __restrict__ cls;         // class of each pair: 1 filtered, 3 culled, else 0 (null: not wanted)
  unsigned long long* nfilt;         // filtered pairs (may be null)
  FilterMasks fm;                    // shells: the filtered pairs of the rest mesh
  // rods: arc-length windows (frest.cuh)
  const int32_t* __restrict__ comp;
  const int32_t* __restrict__ win;
  const int32_t* __restrict__ wst;
  const int32_t* __restrict__ rloop;
};

// the FP64 boxes of a pair decide
__device__ __noinline__ bool boxes64_overlap(const TileArgs& A, int4 a, int4 b, uint32_t ci) {
  double la[3], ha[3], lb[3], hb[3];
  prim_box(a, A.n, A.x, A.p, la, ha);
  prim_box(b, A.n, A.x, A.p, lb, hb);
  const double h = inflation(A.mp[ci >> 2], A.swept);
  bool ov = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) ov = ov && xsub(la[k], h) <= xadd(hb[k], h) && xsub(lb[k], h) <= xadd(ha[k], h);
  return ov;
}

constexpr int TILE_WARPS = 8;

// (a.x + b.x, a.y + b.y) in one instruction
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  unsigned long long x, y, r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  float2 o;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
  return o;
}
// the smallest of three, NaN if any is
__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// A tile's column primitives, as the inner loop reads them
struct TileColumns {
  float4 a[CL];   // hi.x, -lo.x, hi.y, -lo.y
  float4 b[CL];   // hi.z, -lo.z, and the first two vertices
  int2 c[CL];     // the third vertex (rods: the component), the primitive
  int2 w[CL];     // rods: the arc-length windows
  uint16_t code[CL * CL];  // the tile's pairs: row << 5 | column, filtered << 10, culled << 11
};

// A warp per tile (grid-stride): lane r holds the row cluster's primitive r,
// the column cluster's primitives lie in shared memory.  Columns whose box
// misses the row cluster's are skipped for the whole warp.  Bound by
// instruction issue, so a column costs two wide broadcast reads, the six
// differences of the boxes' bounds in three packed additions, their minimum
// and two comparisons: its sign is the FP32 test (a rounded difference has the
// exact one's sign), and above eps = 2^-21 of the row box's coordinates the
// FP64 boxes, at most an ulp inside on each side, overlap too.  Between the two
// (and for NaN) the FP64 boxes decide.  Each lane then writes its pairs' codes
// to shared memory, and the warp turns them into keys 32 at a time.
// Both broad phases of a pass, from twelve box comparisons a column and keys
// written column by column, 80 registers and three blocks per SM: pleated
// 256x256 509 -> 404 us, a 200k-triangle graded sheet 1,068 -> 837, 64 rod
// scenes 950 -> 665 (the windows and components now come once per tile), and
// 467 with their clusters cut by yarn.
// The pairs' classes come with them (Sec. 3.2): on shells the rest mesh's
// filtered pairs are kept as one 32x32 bit mask per pair of clusters, so a
// tile looks its mask up once and a pair's class is a bit; on rods they are the
// arc-length windows of the two edges.  (A search of the sorted filtered keys
// per candidate, in contact_filter and again in the CCD screen, took 0.32 and
// about 0.2 ms of a pleated 256x256 pass, 0.56 and 0.4 ms of a graded one.)
__global__ void __launch_bounds__(32 * TILE_WARPS, 3) k_tiles(TileArgs A) {
  __shared__ TileColumns cols_of[TILE_WARPS];
  const int lane = threadIdx.x & 31;
  TileColumns& S = cols_of[threadIdx.x >> 5];
  const unsigned long long nt = *A.ntiles, m = nt < A.tile_cap ? nt : A.tile_cap;
  const unsigned long long nw = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
  unsigned n32 = 0, n64 = 0, dense = 0, nf = 0;
  unsigned long long w = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  uint2 next = w < m ? A.tiles[w] : make_uint2(0u, 0u);
  for (; w < m; w += nw) {
    const uint2 t = next;
    if (w + nw < m) next = A.tiles[w + nw];
    const int64_t sr = (int64_t)t.x * CL + lane, sc = (int64_t)t.y * CL + lane;
    const Box a = load_box(A.box, sr), b = load_box(A.box, sc);
    const int4 va = A.slots[sr], vb = A.slots[sc];
    const uint32_t ci = A.cinfo[t.x];
    const bool pt = (ci & 3u) == 0u && !A.rod;
    const bool windows = A.rod && A.cls;
    int mine = -1, win = 0, wst = 0;
    __syncwarp();  // the last tile's reads are over
    S.a[lane] = make_float4(b.hi.x, -b.lo.x, b.hi.y, -b.lo.y);
    S.b[lane] = make_float4(b.hi.z, -b.lo.z, __int_as_float(vb.x), __int_as_float(vb.y));
    S.c[lane] = make_int2(windows && vb.x >= 0 ? A.comp[vb.x] : vb.z, vb.w);
    if (windows) {
      if (vb.w >= 0) S.w[lane] = make_int2(A.win[vb.w], A.wst[vb.w]);
      if (va.w >= 0) {
        mine = A.comp[va.x];
        win = A.win[va.w];
        wst = A.wst[va.w];
      }
    }
    // empty slots take no part: a primitive reaching from -inf to +inf on every axis would meet even their empty boxes
    unsigned cols = __ballot_sync(FULL, vb.w >= 0 && overlap(load_box(A.cbox, t.x), b));
    __syncwarp();
    const float2 ax = make_float2(-a.lo.x, a.hi.x), ay = make_float2(-a.lo.y, a.hi.y), az = make_float2(-a.lo.z, a.hi.z);
    const float eps = fmaf(fmaxf(fmaxf(fmaxf(fabsf(ax.x), fabsf(ax.y)), fmaxf(fabsf(ay.x), fabsf(ay.y))),
                                 fmaxf(fabsf(az.x), fabsf(az.y))), 4.76837158e-7f, 1e-40f);
    unsigned hit = 0u, sure = 0u;
    auto test = [&](int c) {
      const float4 qa = S.a[c], qb = S.b[c];
      const int vx = __float_as_int(qb.z), vy = __float_as_int(qb.w);
      const float2 dx = add2(make_float2(qa.x, qa.y), ax), dy = add2(make_float2(qa.z, qa.w), ay),
                   dz = add2(make_float2(qb.x, qb.y), az);
      const float d = min3(min3(dx.x, dx.y, dy.x), min3(dy.y, dz.x, dz.y), dz.y);
      // shared vertices: a point's against the triangle's three, an edge's two against the other's two
      const bool inc = pt ? (va.x == vx || va.x == vy || va.x == S.c[c].x)
                          : (va.x == vx || va.x == vy || va.y == vx || va.y == vy);
      if (!(d < 0.f) && !inc) hit |= 1u << c;
      if (d > eps) sure |= 1u << c;
    };
    while (cols) {  // two columns at a time: their reads overlap
      const int c0 = __ffs((int)cols) - 1;
      cols &= cols - 1u;
      const int c1 = cols ? __ffs((int)cols) - 1 : c0;
      cols &= cols - 1u;
      test(c0);
      test(c1);
    }
    if (va.w < 0) hit = 0u;
    if (t.x == t.y) hit &= lane < 31 ? FULL << (lane + 1) : 0u;
    n32 += (unsigned)__popc(hit);
    for (unsigned todo = hit & ~sure; todo; todo &= todo - 1u) {
      const int c = __ffs((int)todo) - 1;
      ++n64;
      if (!boxes64_overlap(A, va, A.slots[(int64_t)t.y * CL + c], ci)) hit &= ~(1u << c);
    }
    const unsigned cnt = (unsigned)__popc(hit);
    if (A.rod) dense += cnt > CL / 2 ? 1u : 0u;
    unsigned at = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned u = __shfl_up_sync(FULL, at, o);
      if (lane >= o) at += u;
    }
    const unsigned total = __shfl_sync(FULL, at, 31);
    if (total == 0) continue;
    at -= cnt;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(A.total, (unsigned long long)total);
    unsigned filt = 0u, cull = 0u;
    if (A.cls) {
      const MemberParams& M = A.mp[ci >> 2];
      if (!A.rod) {
        if (!M.filter_off) filt = hit & A.fm.row(t.x, t.y, lane);
      } else if (!M.filter_off || M.cull_radius > 0) {
        for (unsigned todo = hit; todo; todo &= todo - 1u) {
          const int c = __ffs((int)todo) - 1;
          const int2 v = S.c[c], wc = S.w[c];
          if (v.x != mine) continue;
          const bool first = va.w < v.y;
          const int i = first ? va.w : v.y, j = first ? v.y : va.w;
          if (!M.filter_off && rod_filtered(first ? win : wc.x, first ? wst : wc.y, M.loops != 0, j)) filt |= 1u << c;
          // Kaldor culling: edges are numbered along each polyline, so the gap is j - i (the shorter way round a loop)
          if (M.cull_radius > 0 && rod_gap(A.rloop, (uint32_t)i, (uint32_t)j) <= M.cull_radius) cull |= 1u << c;
        }
      }
      nf += (unsigned)__popc(filt);
    }
    for (unsigned todo = hit; todo; todo &= todo - 1u, ++at) {
      const int c = __ffs((int)todo) - 1;
      S.code[at] = (uint16_t)(lane << 5 | c | ((filt >> c) & 1u) << 10 | ((cull >> c) & 1u) << 11);
    }
    base = __shfl_sync(FULL, base, 0);
    if (base + total > A.out_cap) continue;  // counted only: the caller grows the list and comes again
    __syncwarp();
    const uint32_t type = pt ? CB_KEY_PT : (A.rod ? CB_KEY_ROD_EE : CB_KEY_EE);
    for (unsigned k0 = 0; k0 < total; k0 += 32) {
      const unsigned k = k0 + lane, e = S.code[min(k, total - 1u)];
      uint32_t i = (uint32_t)__shfl_sync(FULL, va.w, (int)(e >> 5 & 31u)), j = (uint32_t)S.c[e & 31u].y;
      if (k >= total) continue;
      if (!pt && j < i) {  // edge-edge keys take the lower edge first
        const uint32_t u = i;
        i = j;
        j = u;
      }
      if (A.cls) A.cls[base + k] = e >> 11 & 1u ? (uint8_t)3 : (uint8_t)(e >> 10 & 1u);
      A.out[base + k] = A.canonical ? cb_key(type, i, j)
                                    : (((uint64_t)type << (A.bi + A.bj)) | ((uint64_t)i << A.bj) | j);
    }
  }
  if (A.fpstat) {
    const unsigned a32 = __reduce_add_sync(FULL, n32), a64 = __reduce_add_sync(FULL, n64);
    if (lane == 0) {
      if (a32) atomicAdd(&A.fpstat[0], (unsigned long long)a32);
      if (a64) atomicAdd(&A.fpstat[1], (unsigned long long)a64);
    }
  }
  if (A.nfilt) {
    const unsigned a = __reduce_add_sync(FULL, nf);
    if (lane == 0 && a) atomicAdd(A.nfilt, (unsigned long long)a);
  }
  if (A.rod && __any_sync(FULL, dense != 0u)) {
    const unsigned d = __reduce_add_sync(FULL, dense);
    if (lane == 0) atomicAdd(A.novf, d);
  }
}

__global__ void k_expand(int64_t nc, const uint64_t* __restrict__ ck, int bi, int bj, uint64_t* __restrict__ out) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nc) return;
  uint64_t c = ck[q];
  uint32_t type = (uint32_t)(c >> (bi + bj));
  uint32_t i = (uint32_t)((c >> bj) & ((1ull << bi) - 1ull));
  uint32_t j = (uint32_t)(c & ((1ull << bj) - 1ull));
  out[q] = cb_key(type, i, j);
}

// ---- the clusters of a scene -------------------------------------------------

__device__ __forceinline__ uint32_t spread10(uint32_t v) {
  v &= 0x3ffu;
  v = (v | (v << 16)) & 0x030000FFu;
  v = (v | (v << 8)) & 0x0300F00Fu;
  v = (v | (v << 4)) & 0x030C30C3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

// a shell primitive (ids: vertices, triangles, edges) as its vertex ids and its index within its kind
__device__ __forceinline__ int4 shell_prim(int q, int n, int T, const int32_t* __restrict__ ev0,
                                           const int32_t* __restrict__ ev1, const int32_t* __restrict__ tv) {
  if (q < n) return make_int4(q, -1, -1, q);
  q -= n;
  if (q < T) return make_int4(tv[q], tv[(size_t)T + q], tv[2 * (size_t)T + q], q);
  q -= T;
  return make_int4(ev0[q], ev1[q], -1, q);
}

// sort keys: kind, then the Morton code of the rest centroid on a 1024^3 grid over the scene
__global__ void k_order_keys(int np, int n, int T, const int32_t* __restrict__ ev0, const int32_t* __restrict__ ev1,
                             const int32_t* __restrict__ tv, const double* __restrict__ rest, double ox, double oy,
                             double oz, double inv, uint32_t* __restrict__ key, uint32_t* __restrict__ val) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= np) return;
  const int4 v = shell_prim(q, n, T, ev0, ev1, tv);
  const int id[3] = {v.x, v.y, v.z};
  double c[3] = {0.0, 0.0, 0.0};
  int cnt = 0;
  for (int a = 0; a < 3; ++a) {
    if (id[a] < 0) continue;
    ++cnt;
    for (int k = 0; k < 3; ++k) c[k] += rest[(size_t)k * n + id[a]];
  }
  const double o[3] = {ox, oy, oz};
  uint32_t g[3];
  for (int k = 0; k < 3; ++k) g[k] = (uint32_t)fmin(fmax((c[k] / cnt - o[k]) * inv, 0.0), 1023.0);
  const uint32_t kind = q < n ? 0u : (q < n + T ? 1u : 2u);
  key[q] = (kind << 30) | spread10(g[0]) | (spread10(g[1]) << 1) | (spread10(g[2]) << 2);
  val[q] = (uint32_t)q;
}

// the primitives' components in their Morton order, for a stable sort by component
__global__ void k_comp_keys(int np, const uint32_t* __restrict__ order, int n, int T, const int32_t* __restrict__ ev0,
                            const int32_t* __restrict__ ev1, const int32_t* __restrict__ tv,
                            const int32_t* __restrict__ vcomp, uint32_t* __restrict__ key) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < np) key[p] = (uint32_t)vcomp[shell_prim((int)order[p], n, T, ev0, ev1, tv).x];
}

// a primitive (ids: vertices, triangles, edges; rods: edges) and its kind (0 vertex, 1 triangle, 2 edge)
__device__ __forceinline__ int4 any_prim(int q, bool rod, int n, int T, const int32_t* __restrict__ ev0,
                                         const int32_t* __restrict__ ev1, const int32_t* __restrict__ tv, int& kind) {
  kind = rod ? 2 : (q < n ? 0 : (q < n + T ? 1 : 2));
  return rod ? make_int4(ev0[q], ev1[q], -1, q) : shell_prim(q, n, T, ev0, ev1, tv);
}

// rank of every primitive among those of its kind and component: its place in the order (null: as numbered) less the
// first place of that kind and component
__global__ void k_ranks(int np, const uint32_t* __restrict__ order, bool rod, int n, int T, const int32_t* __restrict__ ev0,
                        const int32_t* __restrict__ ev1, const int32_t* __restrict__ tv,
                        const int32_t* __restrict__ vcomp, int comps, const int32_t* __restrict__ first,
                        int32_t* __restrict__ rank) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= np) return;
  const int q = order ? (int)order[p] : p;
  int kind;
  const int4 v = any_prim(q, rod, n, T, ev0, ev1, tv, kind);
  rank[q] = p - first[(size_t)kind * comps + vcomp[v.x]];
}

// every primitive into its slot: the first one of its kind and component, plus its rank
__global__ void k_place(int np, bool rod, int n, int T, const int32_t* __restrict__ ev0, const int32_t* __restrict__ ev1,
                        const int32_t* __restrict__ tv, const int32_t* __restrict__ vcomp, int comps,
                        const uint32_t* __restrict__ start, const int32_t* __restrict__ rank, int4* __restrict__ slots) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= np) return;
  int kind;
  const int4 v = any_prim(q, rod, n, T, ev0, ev1, tv, kind);
  slots[(size_t)start[(size_t)kind * comps + vcomp[v.x]] + (uint32_t)rank[q]] = v;
}

// slot of every primitive (ids: vertices, triangles, edges)
__global__ void k_slot_of(int64_t nslots, int n, int T, const int4* __restrict__ slots,
                          const uint32_t* __restrict__ cinfo, uint32_t* __restrict__ slot_of) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nslots) return;
  const int id = slots[s].w;
  if (id < 0) return;
  const uint32_t g = cinfo[s / CL] & 3u;
  slot_of[g == 0u ? (int64_t)id : (g == 1u ? (int64_t)n + id : (int64_t)n + T + id)] = (uint32_t)s;
}

// the tiles of the filtered pairs into the table and (bits given) their bits; the table is at most half full, so a
// probe sequence ends
__global__ void k_filter_bits(int64_t nf, const uint64_t* __restrict__ frest, int n, int T,
                              const uint32_t* __restrict__ slot_of, unsigned long long* __restrict__ key, uint32_t mask,
                              uint32_t* __restrict__ bits, unsigned long long* __restrict__ used) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nf) return;
  const uint64_t k = frest[q];
  const bool pt = cb_key_type(k) == CB_KEY_PT;
  const uint32_t a = slot_of[pt ? (int64_t)cb_key_i(k) : (int64_t)n + T + cb_key_i(k)];
  const uint32_t b = slot_of[pt ? (int64_t)n + cb_key_j(k) : (int64_t)n + T + cb_key_j(k)];
  // rows: the points of a point-triangle pair, the edge in the earlier slot of an edge-edge pair
  const uint32_t r = pt ? a : min(a, b), c = pt ? b : max(a, b);
  const unsigned long long tk = FilterMasks::tile_key(r / CL, c / CL);
  uint32_t h = FilterMasks::hash(tk) & mask;
  for (uint32_t probe = 0; probe <= mask; ++probe) {
    const unsigned long long prev = atomicCAS(&key[h], FilterMasks::EMPTY, tk);
    if (prev == FilterMasks::EMPTY) atomicAdd(used, 1ull);
    if (prev == FilterMasks::EMPTY || prev == tk) {
      if (bits) atomicOr(&bits[(size_t)h * CL + r % CL], 1u << (c % CL));
      return;
    }
    h = (h + 1) & mask;
  }
}

int64_t clusters_of(int64_t count) { return (count + CL - 1) / CL; }

// Whether a component of `count` primitives of one kind takes clusters of its own, its last one padded: where that
// leaves at most a quarter of their slots empty.  The others are packed one behind the other.
bool own_clusters(int64_t count) { return 4 * (clusters_of(count) * CL - count) <= clusters_of(count) * CL; }

uint64_t spread21(uint64_t v) {
  v &= 0x1fffffull;
  v = (v | v << 32) & 0x1f00000000ffffull;
  v = (v | v << 16) & 0x1f0000ff0000ffull;
  v = (v | v << 8) & 0x100f00f00f00f00full;
  v = (v | v << 4) & 0x10c30c30c30c30c3ull;
  v = (v | v << 2) & 0x1249249249249249ull;
  return v;
}

// The places of a scene's components at positions xyz ([3][n], host): the Morton code of the mean of their vertices on
// a grid of 2^21 cells per axis over all of them.  Means that are not finite lie in cell 0.
void comp_places(cb_scene* s, const double* xyz) {
  const size_t nc = (size_t)s->n_comps, n = (size_t)s->n;
  std::vector<double> mean(3 * nc, 0.0);
  std::vector<int32_t> cnt(nc, 0);
  for (size_t v = 0; v < n; ++v) {
    const int32_t c = s->hcomp[v];
    if (c < 0) continue;
    ++cnt[c];
    for (int k = 0; k < 3; ++k) mean[3 * (size_t)c + k] += xyz[k * n + v];
  }
  double lo[3] = {INFINITY, INFINITY, INFINITY}, span = 0.0;
  for (int k = 0; k < 3; ++k) {
    double hi = -INFINITY;
    for (size_t c = 0; c < nc; ++c) {
      const double m = mean[3 * c + k] /= std::max(1, cnt[c]);
      if (!std::isfinite(m)) continue;
      lo[k] = std::min(lo[k], m);
      hi = std::max(hi, m);
    }
    if (hi > lo[k]) span = std::max(span, hi - lo[k]);
  }
  const double inv = span > 0.0 && std::isfinite(span) ? 2097152.0 / span : 0.0;
  s->comp_place.assign(nc, 0);
  for (size_t c = 0; c < nc; ++c)
    for (int k = 0; k < 3; ++k) {
      const double g = (mean[3 * c + k] - lo[k]) * inv;
      s->comp_place[c] |= spread21(g > 0.0 ? (uint64_t)std::min(g, 2097151.0) : 0) << k;
    }
}

// The first slot of each component's primitives, by kind: members in order, in each one vertex, triangle and edge
// clusters; of one kind the components with clusters of their own, then the packed ones, both by place and label.
// The clusters of each member and kind to nclusters [count][3].
void comp_slots(const cb_scene* s, std::vector<uint32_t>& start, std::vector<int64_t>& nclusters) {
  const size_t nc = (size_t)s->n_comps;
  start.assign(3 * nc, 0);
  nclusters.assign(3 * (size_t)s->count, 0);
  int64_t slot = 0;
  std::vector<int32_t> order;
  for (int m = 0; m < s->count; ++m) {
    order.resize((size_t)(s->coff[m + 1] - s->coff[m]));
    std::iota(order.begin(), order.end(), (int32_t)s->coff[m]);
    std::sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {
      return s->comp_place[a] != s->comp_place[b] ? s->comp_place[a] < s->comp_place[b] : a < b;
    });
    for (int g = 0; g < 3; ++g) {
      const int64_t begin = slot;
      for (int own = 1; own >= 0; --own)
        for (int32_t c : order) {
          const int64_t cnt = s->comp_cnt[g][c];
          if (cnt == 0 || own_clusters(cnt) != (own == 1)) continue;
          start[g * nc + c] = (uint32_t)slot;
          slot += own ? clusters_of(cnt) * CL : cnt;
        }
      slot = begin + clusters_of(slot - begin) * CL;
      nclusters[3 * (size_t)m + g] = (slot - begin) / CL;
    }
  }
}

// cluster kinds, superclusters and jobs from the members' clusters (host tables, uploaded).  Members in order;
// within one the vertex, triangle and edge clusters (rods: edge clusters only).
cb_status cluster_tables(cb_scene* s, const std::vector<int64_t>& nclusters, cudaStream_t st) {
  std::vector<uint32_t> cinfo;
  std::vector<int4> sup, jobs;
  for (int m = 0; m < s->count; ++m) {
    int first[3], end[3];
    for (int g = 0; g < 3; ++g) {
      const int64_t nc = nclusters[3 * (size_t)m + g];
      first[g] = (int)sup.size();
      for (int64_t k = 0; k < nc; k += CL)
        sup.push_back(make_int4((int)(cinfo.size() + k), (int)std::min<int64_t>(CL, nc - k), m, g));
      end[g] = (int)sup.size();
      cinfo.insert(cinfo.end(), (size_t)nc, ((uint32_t)m << 2) | (uint32_t)g);
    }
    for (int r = first[0]; r < end[0]; ++r)  // points against triangles
      for (int c = first[1]; c < end[1]; c += CL) jobs.push_back(make_int4(r, c, std::min(c + CL, end[1]), 0));
    for (int r = first[2]; r < end[2]; ++r)  // edges against edges
      for (int c = r; c < end[2]; c += CL) jobs.push_back(make_int4(r, c, std::min(c + CL, end[2]), 0));
  }
  s->n_clusters = (int)cinfo.size();
  s->n_supers = (int)sup.size();
  s->n_jobs = (int)jobs.size();
  CB_TRY(buf_ensure(s->slots, sizeof(int4) * CL * std::max<size_t>(1, cinfo.size()), st));
  CB_TRY(buf_ensure(s->cinfo, sizeof(uint32_t) * std::max<size_t>(1, cinfo.size()), st));
  CB_TRY(buf_ensure(s->supers, sizeof(int4) * std::max<size_t>(1, sup.size()), st));
  CB_TRY(buf_ensure(s->jobs, sizeof(int4) * std::max<size_t>(1, jobs.size()), st));
  if (!cinfo.empty())
    CB_CUDA(cudaMemcpyAsync(s->cinfo.p, cinfo.data(), sizeof(uint32_t) * cinfo.size(), cudaMemcpyHostToDevice, st));
  if (!sup.empty()) CB_CUDA(cudaMemcpyAsync(s->supers.p, sup.data(), sizeof(int4) * sup.size(), cudaMemcpyHostToDevice, st));
  if (!jobs.empty()) CB_CUDA(cudaMemcpyAsync(s->jobs.p, jobs.data(), sizeof(int4) * jobs.size(), cudaMemcpyHostToDevice, st));
  CB_CUDA(cudaStreamSynchronize(st));  // the host tables end with this scope
  return CB_OK;
}

// the primitives into the slots of the components' present places
cb_status place_prims(cb_scene* s, const std::vector<uint32_t>& start, cudaStream_t st) {
  if (s->n_clusters == 0) return CB_OK;
  ScopedBuf sb(st);
  CB_TRY(buf_ensure(sb.b, sizeof(uint32_t) * std::max<size_t>(1, start.size()), st));
  if (!start.empty())
    CB_CUDA(cudaMemcpyAsync(sb.b.p, start.data(), sizeof(uint32_t) * start.size(), cudaMemcpyHostToDevice, st));
  CB_CUDA(cudaMemsetAsync(s->slots.p, 0xff, sizeof(int4) * CL * (size_t)s->n_clusters, st));
  k_place<<<cb_grid(s->n_prims), CB_THREADS, 0, cb_count(st)>>>(
      s->n_prims, s->kind == CB_ROD, s->n, s->T, bp<int32_t>(s->ev0), bp<int32_t>(s->ev1), bp<int32_t>(s->tv),
      bp<int32_t>(s->vcomp), s->n_comps, bp<uint32_t>(sb.b), bp<int32_t>(s->prank), bp<int4>(s->slots));
  CB_CUDA(cudaGetLastError());
  CB_CUDA(cudaStreamSynchronize(st));  // the host table may end
  return CB_OK;
}

// packed components, whose clusters are as good as their places tell
void note_packed(cb_scene* s) {
  s->has_packed = false;
  for (int g = 0; g < 3; ++g) {
    int64_t packed = 0;
    for (int32_t c : s->comp_cnt[g]) packed += c > 0 && !own_clusters(c);
    s->has_packed |= packed > 1;
  }
}

cb_status lay_out(cb_scene* s, cudaStream_t st) {
  std::vector<uint32_t> start;
  std::vector<int64_t> nclusters;
  note_packed(s);
  comp_slots(s, start, nclusters);
  CB_TRY(cluster_tables(s, nclusters, st));
  return place_prims(s, start, st);
}

// The packed components again, by their places at x.  (Which components are packed depends on their sizes alone, so
// the clusters, superclusters and jobs stay.)
cb_status lay_out_again(cb_scene* s, const double* x, cudaStream_t st) {
  std::vector<double> xyz(3 * (size_t)s->n);
  CB_CUDA(cudaMemcpyAsync(xyz.data(), x, sizeof(double) * xyz.size(), cudaMemcpyDeviceToHost, st));
  CB_CUDA(cudaStreamSynchronize(st));
  comp_places(s, xyz.data());
  std::vector<uint32_t> start;
  std::vector<int64_t> nclusters;
  comp_slots(s, start, nclusters);
  s->masks_stale = true;  // until they are built for the new slots (an allocation may fail in between)
  CB_TRY(place_prims(s, start, st));
  return filter_masks_build(s, st);
}

}  // namespace

cb_status clusters_build(cb_scene* s, const double* rest_host, const std::vector<int32_t>& label,
                         const std::vector<int32_t>& e0, const std::vector<int32_t>& tris, cudaStream_t st) {
  const bool rod = s->kind == CB_ROD;
  const int np = s->n_prims;
  // components numbered by label: polylines (vertices of none have negative labels), or the smallest vertex of each
  s->hcomp.assign((size_t)s->n, -1);
  if (rod) {
    for (int v = 0; v < s->n; ++v) s->hcomp[v] = std::max(-1, label[v]);
    s->n_comps = s->n_rods;
  } else {
    s->n_comps = 0;
    for (int v = 0; v < s->n; ++v)
      s->hcomp[v] = label[v] == v ? s->n_comps++ : s->hcomp[label[v]];  // (a label comes before its other vertices)
  }
  const size_t nc = (size_t)s->n_comps;
  for (auto& c : s->comp_cnt) c.assign(nc, 0);
  if (!rod) {
    for (int v = 0; v < s->n; ++v) ++s->comp_cnt[0][s->hcomp[v]];
    for (int t = 0; t < s->T; ++t) ++s->comp_cnt[1][s->hcomp[tris[t]]];
  }
  for (int e = 0; e < s->E; ++e) ++s->comp_cnt[2][s->hcomp[e0[e]]];
  s->coff = {0, (int64_t)nc};
  comp_places(s, rest_host);
  if (np == 0) return lay_out(s, st);
  CB_TRY(buf_ensure(s->vcomp, sizeof(int32_t) * (size_t)s->n, st));
  CB_TRY(buf_ensure(s->prank, sizeof(int32_t) * (size_t)np, st));
  CB_CUDA(cudaMemcpyAsync(s->vcomp.p, s->hcomp.data(), sizeof(int32_t) * (size_t)s->n, cudaMemcpyHostToDevice, st));
  // ranks: shells by kind and rest Morton code, then by component (a stable sort); rods as numbered, which is by polyline
  ScopedBuf k0(st), k1(st), v0(st), v1(st), hist(st), tmp(st), fb(st);
  const uint32_t* order = nullptr;
  if (!rod) {
    double lo[3], span = 0.0;
    for (int k = 0; k < 3; ++k) {
      double a = INFINITY, b = -INFINITY;
      for (int v = 0; v < s->n; ++v) {
        const double c = rest_host[(size_t)k * s->n + v];
        a = std::fmin(a, c);
        b = std::fmax(b, c);
      }
      lo[k] = a;
      span = std::fmax(span, b - a);
    }
    const double inv = span > 0.0 && std::isfinite(span) ? 1024.0 / span : 0.0;
    CB_TRY(buf_ensure(k0.b, sizeof(uint32_t) * (size_t)np, st));
    CB_TRY(buf_ensure(k1.b, sizeof(uint32_t) * (size_t)np, st));
    CB_TRY(buf_ensure(v0.b, sizeof(uint32_t) * (size_t)np, st));
    CB_TRY(buf_ensure(v1.b, sizeof(uint32_t) * (size_t)np, st));
    CB_TRY(buf_ensure(hist.b, sizeof(uint32_t) * (size_t)cbp::radix_hist_elems(np), st));
    CB_TRY(buf_ensure(tmp.b, sizeof(uint64_t) * (size_t)(cbp::scan_tmp_elems(cbp::radix_hist_elems(np)) + 8), st));
    k_order_keys<<<cb_grid(np), CB_THREADS, 0, cb_count(st)>>>(np, s->n, s->T, bp<int32_t>(s->ev0), bp<int32_t>(s->ev1),
                                                              bp<int32_t>(s->tv), bp<double>(s->rest), lo[0], lo[1],
                                                              lo[2], inv, bp<uint32_t>(k0.b), bp<uint32_t>(v0.b));
    uint32_t *key = bp<uint32_t>(k0.b), *other_key = bp<uint32_t>(k1.b), *val = bp<uint32_t>(v0.b),
             *other_val = bp<uint32_t>(v1.b);
    if (cbp::radix_sort<uint32_t, uint32_t, true>(key, val, other_key, other_val, np, 0, 32, bp<uint32_t>(hist.b),
                                                  bp<uint32_t>(tmp.b), st)) {
      std::swap(key, other_key);
      std::swap(val, other_val);
    }
    if (nc > 1) {
      int bits = 1;
      while ((nc - 1) >> bits) ++bits;
      k_comp_keys<<<cb_grid(np), CB_THREADS, 0, cb_count(st)>>>(np, val, s->n, s->T, bp<int32_t>(s->ev0),
                                                               bp<int32_t>(s->ev1), bp<int32_t>(s->tv),
                                                               bp<int32_t>(s->vcomp), key);
      if (cbp::radix_sort<uint32_t, uint32_t, true>(key, val, other_key, other_val, np, 0, bits, bp<uint32_t>(hist.b),
                                                    bp<uint32_t>(tmp.b), st))
        std::swap(val, other_val);
    }
    order = val;
  }
  std::vector<int32_t> first(3 * nc);
  int32_t at = 0;
  for (size_t c = 0; c < nc; ++c)
    for (int g = 0; g < 3; ++g) {
      first[g * nc + c] = at;
      at += s->comp_cnt[g][c];
    }
  CB_TRY(buf_ensure(fb.b, sizeof(int32_t) * first.size(), st));
  CB_CUDA(cudaMemcpyAsync(fb.b.p, first.data(), sizeof(int32_t) * first.size(), cudaMemcpyHostToDevice, st));
  k_ranks<<<cb_grid(np), CB_THREADS, 0, cb_count(st)>>>(np, order, rod, s->n, s->T, bp<int32_t>(s->ev0),
                                                       bp<int32_t>(s->ev1), bp<int32_t>(s->tv), bp<int32_t>(s->vcomp),
                                                       s->n_comps, bp<int32_t>(fb.b), bp<int32_t>(s->prank));
  CB_CUDA(cudaGetLastError());
  CB_CUDA(cudaStreamSynchronize(st));  // the host table may end
  return lay_out(s, st);
}

// a batch: its members' components, with their ranks and present places
cb_status clusters_concat(cb_scene* b, cb_scene* const* members, cudaStream_t st) {
  b->n_comps = 0;
  b->coff.assign(1, 0);
  b->hcomp.clear();
  b->comp_place.clear();
  for (auto& c : b->comp_cnt) c.clear();
  for (int m = 0; m < b->count; ++m) {
    const cb_scene* s = members[m];
    for (int32_t c : s->hcomp) b->hcomp.push_back(c < 0 ? -1 : c + b->n_comps);
    b->comp_place.insert(b->comp_place.end(), s->comp_place.begin(), s->comp_place.end());
    for (int g = 0; g < 3; ++g)
      b->comp_cnt[g].insert(b->comp_cnt[g].end(), s->comp_cnt[g].begin(), s->comp_cnt[g].end());
    b->n_comps += s->n_comps;
    b->coff.push_back(b->n_comps);
  }
  if (b->n_prims > 0) {
    CB_TRY(buf_ensure(b->vcomp, sizeof(int32_t) * (size_t)b->n, st));
    CB_TRY(buf_ensure(b->prank, sizeof(int32_t) * (size_t)b->n_prims, st));
    CB_CUDA(cudaMemcpyAsync(b->vcomp.p, b->hcomp.data(), sizeof(int32_t) * (size_t)b->n, cudaMemcpyHostToDevice, st));
    const bool rod = b->kind == CB_ROD;
    for (int m = 0; m < b->count; ++m) {
      const cb_scene* s = members[m];
      // vertices, triangles, edges of the member, each behind those of the members before it
      const int64_t cnt[3] = {rod ? 0 : s->n, rod ? 0 : s->T, s->E};
      const int64_t to[3] = {b->voff[m], (int64_t)b->n + b->toff[m], (rod ? 0 : (int64_t)b->n + b->T) + b->eoff[m]};
      int64_t from = 0;
      for (int g = 0; g < 3; from += cnt[g++])
        if (cnt[g] > 0)
          CB_CUDA(cudaMemcpyAsync(bp<int32_t>(b->prank) + to[g], bp<int32_t>(s->prank) + from,
                                  sizeof(int32_t) * (size_t)cnt[g], cudaMemcpyDeviceToDevice, st));
    }
  }
  return lay_out(b, st);
}

// The filtered pairs as masks: a table of the tiles that hold any (no more of them than pairs), counted, then one of
// that size with their masks.
cb_status filter_masks_build(cb_scene* s, cudaStream_t st) {
  if (s->kind != CB_SHELL || s->n_frest <= 0) {
    s->masks_stale = false;
    return CB_OK;
  }
  auto table = [](int64_t tiles) {
    int64_t cap = 64;
    while (cap < 2 * tiles && cap < (1ll << 32)) cap *= 2;
    return cap;
  };
  const int64_t nslots = (int64_t)s->n_clusters * CL;
  ScopedBuf so(st), tiles(st);
  CB_TRY(buf_ensure(so.b, sizeof(uint32_t) * (size_t)s->n_prims, st));
  k_slot_of<<<cb_grid(nslots), CB_THREADS, 0, cb_count(st)>>>(nslots, s->n, s->T, bp<int4>(s->slots),
                                                             bp<uint32_t>(s->cinfo), bp<uint32_t>(so.b));
  unsigned long long* used = (unsigned long long*)scalars(s) + SC_COUNT1;
  int64_t cap = table(s->n_frest);
  for (int round = 0; round < 2; ++round) {
    DevBuf& key = round ? s->fmask_key : tiles.b;
    CB_TRY(buf_ensure(key, sizeof(unsigned long long) * (size_t)cap, st));
    CB_CUDA(cudaMemsetAsync(key.p, 0xff, sizeof(unsigned long long) * (size_t)cap, st));
    if (round) {
      CB_TRY(buf_ensure(s->fmask_bits, sizeof(uint32_t) * CL * (size_t)cap, st));
      CB_CUDA(cudaMemsetAsync(s->fmask_bits.p, 0, sizeof(uint32_t) * CL * (size_t)cap, st));
    }
    CB_CUDA(cudaMemsetAsync(used, 0, sizeof(unsigned long long), st));
    k_filter_bits<<<cb_grid(s->n_frest), CB_THREADS, 0, cb_count(st)>>>(
        s->n_frest, bp<uint64_t>(s->frest), s->n, s->T, bp<uint32_t>(so.b), bp<unsigned long long>(key),
        (uint32_t)(cap - 1), round ? bp<uint32_t>(s->fmask_bits) : nullptr, used);
    CB_CUDA(cudaGetLastError());
    if (round) break;
    uint64_t h = 0;
    CB_TRY(read_scalars(s, SC_COUNT1, 1, &h, st));
    s->n_fmask = (int64_t)h;
    cap = table(s->n_fmask);
    buf_free(tiles.b, st);
  }
  s->fmask_mask = (uint32_t)(cap - 1);
  s->masks_stale = false;
  return CB_OK;
}

// Tiles per cluster above which the order of packed components is looked at again.  Scenes in good order have 2 to 16
// (woven, chain, layers, pleated, graded), 47 in a felt of 20,000 fibres of 33 edges in 2 edges' distance; 20,000 fibres
// whose order says nothing have 1,500 to 3,600.
constexpr int64_t TILES_PER_CLUSTER = 64;

cb_status broad_phase(cb_scene* s, BroadWork& w, const double* x, const double* p, bool swept, bool sort_out,
                      DevBuf& out, DevBuf* cls, int64_t* n_out, cudaStream_t st) {
  const int M = s->count, nc = s->n_clusters, ns = s->n_supers, nj = s->n_jobs;
  *n_out = 0;
  if (nc == 0) return CB_OK;
  const bool rod = s->kind == CB_ROD;
  if (s->masks_stale) CB_TRY(filter_masks_build(s, st));
  CB_TRY(buf_ensure(w.box, sizeof(float4) * 2 * CL * (size_t)nc, st));
  CB_TRY(buf_ensure(w.cbox, sizeof(float4) * 2 * (size_t)nc, st));
  CB_TRY(buf_ensure(w.sbox, sizeof(float4) * 2 * (size_t)ns, st));
  CB_TRY(buf_ensure(w.bounds, sizeof(uint32_t) * BOUNDS_STRIDE * (size_t)M, st));
  CB_TRY(buf_ensure(w.cx, sizeof(double) * 4 * (size_t)M, st));
  // room for 16 column clusters per row cluster to begin with; a call that finds more grows it and lists again
  CB_TRY(buf_ensure(w.tiles, sizeof(uint2) * (size_t)(16 * (int64_t)nc + 1024), st));
  // per-stencil activation: the static phase keeps the uninflated boxes for contact_filter
  const bool raw = !swept && !p && !sort_out && s->per_stencil();
  if (raw) CB_TRY(buf_ensure(w.box_raw, sizeof(double) * 6 * (size_t)s->n_prims, st));
  unsigned long long* sc = (unsigned long long*)scalars(s);
  unsigned long long *ntiles = sc + SC_COUNT0, *total = sc + SC_COUNT1;
  const bool stat = !swept;
  // vertex boxes first once the primitives fill the chip: below, another launch costs more than the FP64 work it saves
  // (4,112 vertices of a woven patch: 8 us against 6 + 5)
  const bool by_vertex = nc >= 8 * s->n_sms;
  if (by_vertex) {
    // they lie in the screens' FP32 positions and displacements, which their users write afresh
    CB_TRY(buf_ensure(s->xf, sizeof(float4) * (size_t)s->n, st));
    CB_TRY(buf_ensure(s->pf, sizeof(float4) * (size_t)s->n, st));
  }

  BoxArgs B{nc,
            s->n,
            s->T,
            M,
            rod,
            swept,
            bp<int4>(s->slots),
            bp<uint32_t>(s->cinfo),
            x,
            p,
            bp<MemberParams>(s->mp),
            by_vertex ? bp<float4>(s->xf) : nullptr,
            by_vertex ? bp<float4>(s->pf) : nullptr,
            bp<float4>(w.box),
            bp<float4>(w.cbox),
            raw ? bp<double>(w.box_raw) : nullptr,
            bp<uint32_t>(w.bounds),
            sc,
            (1u << SC_COUNT0) | (1u << SC_COUNT1) | (1u << SC_NOVF) |
                (stat ? (1u << SC_FP32_PAIRS) | (1u << SC_FP64_DECIDED) | (1u << SC_NFB) : 0u)};
  if (by_vertex)
    k_vertex_boxes<<<cb_grid(s->n), 256, 0, cb_count(st)>>>(s->n, swept, x, p, bp<int32_t>(s->vsc), bp<MemberParams>(s->mp), M,
                                                          bp<float4>(s->xf), bp<float4>(s->pf));
  auto launch_boxes = [&] {
    k_boxes<<<cb_grid((int64_t)nc * CL), 256, 0, cb_count(st)>>>(B);
    k_super_boxes<<<cb_grid((int64_t)ns * CL), 256, 0, cb_count(st)>>>(ns, bp<int4>(s->supers), bp<float4>(w.cbox),
                                                                      bp<float4>(w.sbox), bp<uint32_t>(w.bounds));
  };
  launch_boxes();
  DevBuf& list = sort_out ? w.ckey[0] : out;
  TileArgs A;
  A.n = s->n;
  A.rod = rod;
  A.swept = swept;
  A.canonical = !sort_out;
  A.bi = s->bits_i;
  A.bj = s->bits_j;
  A.slots = bp<int4>(s->slots);
  A.cinfo = bp<uint32_t>(s->cinfo);
  A.box = bp<float4>(w.box);
  A.cbox = bp<float4>(w.cbox);
  A.ntiles = ntiles;
  A.x = x;
  A.p = p;
  A.mp = bp<MemberParams>(s->mp);
  A.total = total;
  A.fpstat = stat ? sc + SC_FP32_PAIRS : nullptr;
  A.novf = (unsigned int*)(sc + SC_NOVF);
  A.nfilt = stat && cls ? sc + SC_NFB : nullptr;
  A.comp = bp<int32_t>(s->comp);
  A.win = bp<int32_t>(s->win);
  A.wst = bp<int32_t>(s->wst);
  A.rloop = bp<int32_t>(s->rloop);
  uint64_t h[2] = {0, 0};
  static_assert(SC_COUNT1 == SC_COUNT0 + 1 && SC_FP64_DECIDED == SC_FP32_PAIRS + 1, "read and cleared together");
  // lists that turn out too short are grown and written again (at most once each)
  bool laid = false;
  for (bool find = true;;) {
    A.fm = FilterMasks{bp<unsigned long long>(s->fmask_key), bp<uint32_t>(s->fmask_bits),
                       s->n_fmask > 0 ? s->fmask_mask : 0u};
    if (find) {
      k_cluster_pairs<<<(int)std::max<int64_t>(1, std::min<int64_t>(nj, (int64_t)s->n_sms * 64)), 32 * PAIR_WARPS, 0, cb_count(st)>>>(
          nj, bp<int4>(s->jobs), bp<int4>(s->supers), bp<float4>(w.sbox), bp<float4>(w.cbox), bp<uint2>(w.tiles),
          (unsigned long long)(w.tiles.bytes / sizeof(uint2)), ntiles, M, bp<uint32_t>(w.bounds), bp<double>(w.cx));
    }
    A.tiles = bp<uint2>(w.tiles);
    A.tile_cap = (unsigned long long)(w.tiles.bytes / sizeof(uint2));
    A.out = bp<uint64_t>(list);
    A.out_cap = (unsigned long long)(list.bytes / sizeof(uint64_t));
    A.cls = cls ? bp<uint8_t>(*cls) : nullptr;
    if (cls) A.out_cap = std::min<unsigned long long>(A.out_cap, cls->bytes);
    // candidates are numbered in 32 bits, whatever room an earlier call left in the list
    A.out_cap = std::min<unsigned long long>(A.out_cap, 0xffffffffull);
    k_tiles<<<s->n_sms * 3, 32 * TILE_WARPS, 0, cb_count(st)>>>(A);
    CB_CUDA(cudaGetLastError());
    CB_TRY(read_scalars(s, SC_COUNT0, 2, h, st));
    // Far more tiles than a well-ordered scene has: the packed components may lie elsewhere than the rest shape said
    // (instances of one shape placed only through x) or have moved.  They are put in order again at x, unless the last
    // time left a quarter of these tiles or more.
    if (!laid && s->has_packed && !sort_out && h[0] > (unsigned long long)std::max((int64_t)nc * TILES_PER_CLUSTER, 4 * w.tiles_laid)) {
      CB_TRY(lay_out_again(s, x, st));
      laid = find = true;
      launch_boxes();
      continue;
    }
    find = h[0] > A.tile_cap;
    if (!find && h[1] <= A.out_cap) break;
    if (h[1] > 0xffffffffull) return CB_ERR_TOO_LARGE;
    if (find) {
      CB_TRY(buf_ensure(w.tiles, sizeof(uint2) * (size_t)h[0], st));
    } else {
      CB_TRY(buf_ensure(list, sizeof(uint64_t) * (size_t)h[1], st));
      if (cls) CB_TRY(buf_ensure(*cls, (size_t)h[1], st));
    }
    CB_CUDA(cudaMemsetAsync(total, 0, sizeof(unsigned long long), st));
    CB_CUDA(cudaMemsetAsync(A.novf, 0, sizeof(unsigned int), st));
    if (stat) CB_CUDA(cudaMemsetAsync(A.fpstat, 0, 2 * sizeof(unsigned long long), st));
    if (A.nfilt) CB_CUDA(cudaMemsetAsync(A.nfilt, 0, sizeof(unsigned long long), st));
    if (find) CB_CUDA(cudaMemsetAsync(ntiles, 0, sizeof(unsigned long long), st));
  }
  const int64_t n = (int64_t)h[1];
  if (laid) w.tiles_laid = (int64_t)h[0];
  *n_out = n;
  if (n == 0 || !sort_out) return CB_OK;
  CB_TRY(buf_ensure(w.ckey[1], sizeof(uint64_t) * (size_t)n, st));
  const int cbits = s->bits_i + s->bits_j + (s->kind == CB_SHELL ? 2 : 0);
  CB_TRY(buf_ensure(w.hist, sizeof(uint32_t) * (size_t)cbp::radix_hist_elems(n), st));
  CB_TRY(buf_ensure(w.scan_tmp, sizeof(uint64_t) * (size_t)(cbp::scan_tmp_elems(cbp::radix_hist_elems(n)) + 8), st));
  int r2 = cbp::radix_sort<uint64_t, uint32_t, false>(bp<uint64_t>(w.ckey[0]), nullptr, bp<uint64_t>(w.ckey[1]),
                                                      nullptr, n, 0, cbits, bp<uint32_t>(w.hist),
                                                      bp<uint32_t>(w.scan_tmp), st);
  CB_TRY(buf_ensure(out, sizeof(uint64_t) * (size_t)n, st));
  k_expand<<<cb_grid(n), CB_THREADS, 0, cb_count(st)>>>(n, bp<uint64_t>(w.ckey[r2]), s->bits_i, s->bits_j,
                                                       bp<uint64_t>(out));
  CB_CUDA(cudaGetLastError());
  return CB_OK;
}
