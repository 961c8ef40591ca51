// scene.cuh -- internal scene object and the launchers each stage file provides.
#pragma once
#include <vector>

#include "common.cuh"

// A device buffer remembers the allocator that made it (NULL: the library's
// own stream-ordered pool) and the byte counter of the scene it is charged to.
struct DevBuf {
  void* p = nullptr;
  size_t bytes = 0;
  const cb_allocator* alloc = nullptr;
  int64_t* charged = nullptr;
};

// Where the buffers of the current API call come from: set for the duration
// of each call that may allocate (AllocScope), read by buf_ensure.
struct AllocCtx {
  const cb_allocator* alloc = nullptr;
  int64_t* charged = nullptr;
};
AllocCtx& alloc_ctx();
struct AllocScope {
  AllocCtx saved;
  AllocScope(const cb_allocator* a, int64_t* charged) : saved(alloc_ctx()) {
    alloc_ctx().alloc = a;
    alloc_ctx().charged = charged;
  }
  ~AllocScope() { alloc_ctx() = saved; }
};

// A growable device buffer: keeps its allocation, grows by 25 % headroom.
// Allocates through the current AllocScope's allocator (or the library's
// pool) and charges the scope's counter; frees through the buffer's own
// allocator (after the stream's work is done, since a caller's allocator may
// hand the memory out again at once).
cb_status buf_ensure(DevBuf& b, size_t bytes, cudaStream_t st);
void buf_free(DevBuf& b, cudaStream_t st);

// A device buffer local to one call, released on every way out of its scope
// (error returns included).
struct ScopedBuf {
  DevBuf b;
  cudaStream_t st;
  explicit ScopedBuf(cudaStream_t s) : st(s) {}
  ~ScopedBuf() { buf_free(b, st); }
  ScopedBuf(const ScopedBuf&) = delete;
  ScopedBuf& operator=(const ScopedBuf&) = delete;
};
template <typename T>
static inline T* bp(const DevBuf& b) {
  return (T*)b.p;
}

// Per-member parameters.  A plain scene has one member; a batch (several
// scenes merged into one index space, cb_batch_create) has one per scene.
struct MemberParams {
  double xi, dhat, a, kappa;
  double dbar_min;        // 0 when nothing is filtered
  int32_t single, core_temp, filter_off, n_prims;
  // FP32 copies rounded up, for the screens' rigorous FP32 comparisons (set
  // at upload): a (1 + 1e-9) + 1e-9, dbar_min (1 + 1e-9) + 1e-9,
  // xi (1 + 1e-9) + 1e-9, xi
  float thrU32, thrF32, thrC32, xi32;
  int32_t cull_radius;    // CB_FILTER_KALDOR: rod edge pairs of one polyline this close are culled; else 0
  int32_t per_comp;       // CB_DBAR_PER_COMPONENT: class-F width from dbar_comp by component label
  double dbar_fmax;       // largest class-F width of the member (= dbar_min unless per_comp)
  int32_t loops;          // rods: the member has closed loops (backward arc-length windows to test)
  int32_t mollify;        // CB_EE_MOLLIFIER: edge-edge pairs take IPC's mollifier
  int32_t per_stencil;    // CB_PER_STENCIL: class-F candidates outside their own width are dropped
};

// Workspace of one broad phase (static or swept) -- reused between calls.
struct BroadWork {
  // cb_set_tuning's knobs: kept and returned; the cluster broad phase has no cells to size
  float cell_factor = 1.0f;
  int pair_block = CB_THREADS;
  DevBuf box;         // float4 lo, float4 hi per slot (inflated, rounded outwards)
  DevBuf cbox, sbox;  // ... per cluster and per supercluster
  DevBuf box_raw;     // per-stencil activation (static phase): double lo[3], hi[3] per primitive, not inflated
  DevBuf bounds;      // per member: 6 x uint32 ordered-float min/max
  DevBuf cx;          // per member: double centre[3], X (max |coordinate - centre|)
  DevBuf tiles;       // uint2 pairs of overlapping clusters
  int64_t tiles_laid = 0;  // their number after the clusters were last laid out again for this phase
  DevBuf ckey[2];     // uint64 compact candidate keys (ping-pong; sorted lists only)
  DevBuf scan_tmp;
  DevBuf hist;
};

struct cb_scene {
  // the caller's allocator (copied at create; has_alloc false: the library's pool)
  // and the bytes of device memory the scene holds now
  cb_allocator allocator{};
  bool has_alloc = false;
  int64_t live_bytes = 0;
  const cb_allocator* alloc_ptr() const { return has_alloc ? &allocator : nullptr; }
  int kind = 0;
  int n = 0, E = 0, T = 0, n_rods = 0;
  int n_prims = 0;     // broad-phase primitives
  int bits_i = 0, bits_j = 0;
  double xi = 0, dhat = 0, a = 0, kappa = 1;   // member 0 (plain scenes: the scene)
  int filter = CB_FILTER_DOUBLE;
  int core_temp = 1;
  double dbar_min = 0;  // +inf when nothing is filtered
  // members (1 for a plain scene)
  int count = 1;
  std::vector<MemberParams> hmp;
  DevBuf mp;            // MemberParams [count]
  DevBuf vsc;           // int32 [n] member of each vertex
  std::vector<int64_t> voff, eoff, toff;  // member offsets of vertices, edges, triangles (count+1)
  int64_t n_frest_pt = 0;                 // shells: point-triangle keys at the head of frest
  DevBuf macc;          // per member: double energy, u64 alpha bits, u64 status, double upper bound of alpha
  void* hstage_host = nullptr;  // pinned staging (the largest per-member record x members + 256)
  cudaStream_t last_stream = nullptr;
  int device = 0;
  int n_sms = 152;      // multiprocessors of the device (caps of grid-stride launches: a few blocks per SM)
  int proj_occ = 0;     // resident blocks per SM of k_hess_proj (0: not looked up yet)

  // topology on device
  DevBuf ev0, ev1;      // int32 [E]
  DevBuf tv;            // int32 [3][T]
  DevBuf comp;          // int32 [n]
  DevBuf rest;          // double [3][n]
  DevBuf rod_ptr;       // int32 [n_rods+1] (rods)
  // connected components (rods: polylines), numbered by label, members' ones behind each other
  int n_comps = 0;
  std::vector<int32_t> hcomp;         // [n] component of each vertex (-1: in none)
  std::vector<int32_t> comp_cnt[3];   // their vertices, triangles and edges (rods: edges only)
  std::vector<uint64_t> comp_place;   // their places: Morton code at rest, or at the positions of the last lay_out_again
  std::vector<int64_t> coff;          // member offsets of the components (count + 1)
  bool has_packed = false;            // several components share clusters
  DevBuf vcomp;         // int32 [n] hcomp
  DevBuf prank;         // int32 [n_prims] rank of each primitive among those of its kind and component
  // clusters of 32 primitives and superclusters of 32 clusters (broad.cu)
  int n_clusters = 0, n_supers = 0, n_jobs = 0;
  DevBuf slots;         // int4 [n_clusters][32]: a primitive's vertices (-1: none) and its index within its kind (-1: pad)
  DevBuf cinfo;         // uint32 [n_clusters] member << 2 | kind (0 vertex, 1 triangle, 2 edge)
  DevBuf supers;        // int4: first cluster, count, member, kind
  DevBuf jobs;          // int4: row supercluster, first and end column supercluster (at most 32)
  // filter tables
  DevBuf S;             // double [n] rods: arc length
  DevBuf win;           // int32 [E] rods: last filtered partner edge
  DevBuf wst;           // int32 [E] rods: first partner edge of the backward window on a closed loop (-1: none)
  DevBuf rloop;         // int32 [E] rods: edge count of the edge's closed loop (0: open polyline)
  DevBuf rlast;         // int32 [E] rods: last (closing) edge of the edge's closed loop (-1: open)
  DevBuf elen2;         // double [E] squared rest length of each edge (the mollifier's threshold)
  DevBuf ruv;           // double [3][n] shells: the flat pattern (u, v, 0), when given; reference distances there
  bool geodesic = false;  // shells, CB_DBAR_GEODESIC: reference distances are geodesic distances on the rest mesh
  // ... its mesh adjacency, host copies kept until the rest filter has run: edge of (t_k, t_k+1) [T][3],
  // faces of an edge [E][2] (-1: none), faces around a vertex (CSR [n+1], [3T])
  std::vector<int32_t> geo_te, geo_ef, geo_vfp, geo_vf;
  DevBuf frest;         // uint64 shells: sorted rest-filtered keys
  DevBuf frest_dbar;    // double
  DevBuf dbar_comp;     // uint64 bits of the per-component dbar_min, by component label (n entries)
  double dbar_fmax = 0.0;  // largest per-component dbar_min (finite), or dbar_min
  int64_t n_frest = 0;
  // shells: frest as bit masks over pairs of clusters (frest.cuh, FilterMasks)
  DevBuf fmask_key;     // uint64 [fmask_cap], a power of two
  DevBuf fmask_bits;    // uint32 [fmask_cap][32]
  uint32_t fmask_mask = 0;  // fmask_cap - 1
  bool masks_stale = false;  // the clusters changed and the masks do not fit them yet
  int64_t n_fmask = 0;  // pairs of clusters with filtered pairs

  // pass state
  BroadWork bw;         // static broad phase
  BroadWork bwc;        // swept broad phase (CCD)
  DevBuf cand;          // uint64 [nc] sorted candidate keys
  int64_t n_cand = 0;
  DevBuf klass;         // uint8 [nc]
  DevBuf cand_alt, klass_alt;  // per-stencil activation: the compacted candidates before the swap
  int64_t n_dropped = 0;       // last contact_filter: class-F candidates outside their own width
  bool per_stencil() const {
    for (const MemberParams& m : hmp)
      if (m.per_stencil) return true;
    return false;
  }
  DevBuf cd;            // double [nc] distance
  DevBuf cflag, cpos;   // per-stencil activation: uint32 keep flags of the candidates and their scan
  // ... of the active candidates only: distance (cd), type and final class (with C; | CB_CLS_MOLLIFIED)
  DevBuf ctype;         // int8 [nc]
  DevBuf ccls;          // uint8 [nc]
  DevBuf clist;         // uint32 [nc] candidates of class C, SC_NCORE of them
  bool core_valid = false;  // clist belongs to the current candidates
  int64_t n_active = 0;
  DevBuf aidx;          // uint32 [nc] active candidates, two-ended (pairs.cuh, ActiveList)
  int64_t n_plane = 0, act_cap = 0;
  DevBuf bkey;          // uint2 [16 na] (row, column) of the active stencils' blocks, distinct within a run
  DevBuf rcol;          // uint32 [16 na] their columns, bucketed by row
  DevBuf bsr_row;       // int32 [n+1]
  DevBuf bsr_col;       // int32 [nnzb]
  DevBuf bsr_val;       // double [nnzb][9]
  DevBuf row_cnt;       // uint32 [5][n+1]: keys, fill cursor, distinct columns and bucket offset of each row; long rows
                        // (from k_row_unique_long on: the first two the rows past ROW_BLOCK_MAX and their first entries)
  DevBuf hkey, hflag, hhist;  // rows past ROW_BLOCK_MAX (narrow.cu): uint64 keys, uint32 flags and positions, digit counts
  int64_t nnzb = 0;
  DevBuf mlist;         // uint32 [nc] active candidates with a mollifier below 1 (CB_EE_MOLLIFIER)
  DevBuf hB9;           // CB_EE_MOLLIFIER: queued reduced Hessians (packed, element-major)
  DevBuf xf, pf;         // float [3][n]: centred FP32 copies of x and of p
  DevBuf dlist;          // uint32: candidates / CCD pairs queued for the FP64 phase
  DevBuf ccd_keys;      // uint64 [nccd]
  DevBuf ccd_t;         // double [nccd] t_p or a lower bound of it; not written where the class byte has CB_CCD_ONE
  DevBuf ccd_cls;       // uint8 [nccd] class | CB_CCD_EXACT when t is exact | CB_CCD_ONE when it is 1
  DevBuf ccd_list;      // uint32 pairs left for the FP64 iteration
  DevBuf ccd_ulist;     // uint32 pairs still unresolved after the first-step pass
  int64_t n_ccd = 0;
  // lagged friction (friction_lag / friction_eval / friction_spmv)
  DevBuf fr_key;        // uint64 [nf] keys of the lagged pairs
  DevBuf fr_st;         // int4 [nf] their stencil vertices
  DevBuf fr_dat;        // double [8][nf]: lambda, beta[4], n[3] (element-major)
  DevBuf fr_hw;         // double [6][nf]: packed tangent Hessian (xx xy xz yy yz zz) of the last friction_eval
  int64_t n_fric = 0;
  double fr_mu = 0.0, fr_eps = 0.0;
  bool fr_lagged = false, fr_hw_valid = false;
  DevBuf scan_tmp;
  DevBuf dev_scalars;   // misc device scalars (counters, energy, alpha bits, status)

  uint64_t* h_pinned = nullptr;  // pinned host scratch (64 slots)
  int32_t status_host = 0;

  bool timing = false;
  // stage events: [2k, 2k+1] around stage k of cb_get_stage_ms, [10, 11] around
  // the Hessian kernels, [12] the end of stage (c) inside barrier_eval (the
  // active count known); cd_split: the last barrier_eval recorded [12]
  cudaEvent_t ev[13] = {};
  bool cd_split = false;
  float stage_ms[5] = {0, 0, 0, 0, 0};
  int64_t counts_filtered = 0, counts_core = 0;
  int ccd_max_iters = 0;
};

// device scalar slots (uint64 each) inside dev_scalars
enum {
  SC_COUNT0 = 0,
  SC_COUNT1 = 1,
  SC_STATUS = 2,
  SC_ENERGY = 3,
  SC_ALPHA_BITS = 4,
  SC_DBAR_MIN_BITS = 5,
  SC_ITERS = 6,
  SC_NFILT = 7,
  SC_NCORE = 8,
  SC_N9 = 9,
  SC_N6 = 10,
  SC_NLIST = 11,        // two uint32 counters: point-triangle and edge-edge pairs for the exact distance
  SC_N4 = 14,           // point-edge pairs (but for SC_N6's)
  SC_NU = 15,           // CCD pairs left unresolved by the first step
  SC_FP32_PAIRS = 12,   // broad phase of contact_build: pairs passing the FP32 box test
  SC_FP64_DECIDED = 13, // ... of which the FP64 boxes decided
  SC_KSPLIT = 16,       // two uint32 counters: face / line-line pairs, the other active pairs
  SC_NOVF = 17,         // broad phase: rod rows with more than half of a cluster as partners
  SC_NBK = 18,          // BSR pattern: keys left by the runs of k_block_keys
  SC_FETCH = 19,        // ccd_step, FP64 iteration: pairs of the list handed out so far
  SC_NMOLL = 20,        // barrier_eval: mollified edge-edge pairs
  SC_GEO_COUNT = 21,    // geodesic rest filter: (edge, vertex) entries below the activation
  SC_GEO_ERR = 22,      // ... error bits of its sources (a fixed capacity exceeded)
  SC_NX = 23,           // ccd_step: two uint32 counters, point-triangle and edge-edge pairs of the FP64 iteration
  SC_NLONG = 24,        // barrier_eval: rows of the pattern with buckets past a warp's
  SC_NFB = 25,          // contact_build: filtered pairs among the candidates
  SC_HUGE = 26,         // barrier_eval: rows of the pattern with buckets past a block's << 32 | their entries
  SC_N = 27
};
// read_scalars stages up to SC_N scalars through the pinned host scratch
static_assert(SC_N <= 32, "the scalars must fit the pinned scratch and a 32-bit mask");

static inline uint64_t* scalars(cb_scene* s) { return (uint64_t*)s->dev_scalars.p; }

// per-member accumulator slots (uint64 / double each) inside macc
enum { MACC_E = 0, MACC_ALPHA = 1, MACC_STATUS = 2, MACC_HI = 3, MACC_STRIDE = 4 };
// flags of a CCD pair's class byte: t_p is exact (else ccd_t holds a lower bound), and it is 1
constexpr uint8_t CB_CCD_EXACT = 0x80, CB_CCD_ONE = 0x40;

// read n uint64 device scalars into host (sync on stream)
cb_status read_scalars(cb_scene* s, int first, int count, uint64_t* out, cudaStream_t st);

// broad.cu
// The clusters of a new scene (topology and rest positions on the device; on
// the host the same positions, the vertices' component labels, the edges'
// first vertices and the triangles) or of a batch (of its members' components).
cb_status clusters_build(cb_scene* s, const double* rest_host, const std::vector<int32_t>& label,
                         const std::vector<int32_t>& e0, const std::vector<int32_t>& tris, cudaStream_t st);
cb_status clusters_concat(cb_scene* b, cb_scene* const* members, cudaStream_t st);
// Candidate pairs of x (p == nullptr) or of the sweep x -> x + p.  Boxes are
// inflated per member by a/2 (static) or xi/2 (swept = true).  Writes the
// canonical keys into *out (grown as needed), in ascending order when
// sort_out is set and otherwise in tile order, their classes (1 filtered,
// 3 culled, else 0) into *cls unless null, and their count into *n_out.
cb_status broad_phase(cb_scene* s, BroadWork& w, const double* x, const double* p, bool swept, bool sort_out,
                      DevBuf& out, DevBuf* cls, int64_t* n_out, cudaStream_t st);
// the bit masks of the filtered pairs s->frest
cb_status filter_masks_build(cb_scene* s, cudaStream_t st);

// narrow.cu
cb_status filter_precompute(cb_scene* s, cudaStream_t st);
// geodesic.cu: the rest filter's flag / dbar / minima of the rest-broad-phase
// candidates with geodesic reference distances (CB_DBAR_GEODESIC)
cb_status geo_rest_dbar(cb_scene* s, const uint64_t* cand, int64_t nc, uint32_t* flag, double* dbar,
                        unsigned long long* dmin, unsigned long long* dcomp, cudaStream_t st);
cb_status filter_apply(cb_scene* s, cudaStream_t st);
// energy_only: distances and energy (no active list, gradient, Hessian or BSR)
cb_status barrier_run(cb_scene* s, const double* x, double* energy, double* grad, bool energy_only,
                      cudaStream_t st);

// ccd.cu
cb_status ccd_run(cb_scene* s, const double* x, const double* p, double* alpha, cudaStream_t st);

// narrow.cu: FP32 copy of (v - centre of the vertex's member) (cx null: no centring)
cb_status to_f32(cb_scene* s, const double* v, const double* cx, DevBuf& out, cudaStream_t st);
