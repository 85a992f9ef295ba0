// k_trace.cu -- ray casting against a scene of animated sparse voxel octrees.
//
// Per ray (Espe et al., Sec. III-IV):
//   * instance culling: conservative ray / bounding-sphere tests (Eq. 4 in its
//     general form, |d| != 1) against the cluster spheres, then the part
//     spheres of the clusters that are hit (warp vote skips a cluster no lane
//     needs);
//   * depth sorting: candidate parts are visited in increasing sphere entry t
//     and the walk stops once the best hit lies before the next entry
//     (Sec. IV-B);
//   * per candidate part: the ray is moved into the part's frame by the
//     inverse pose (Eq. 2-3; d is not renormalised, so t is shared by all
//     parts) and an iterative front-to-back octree descent runs over the
//     child-descriptor nodes;
//   * closest hit (t, part, voxel), ties broken by smaller part, then voxel.
//
// FP32 certification.  Every FP32 slab test runs on boxes inflated (and, at
// leaves, also deflated) by eta, a per (ray, part) bound on the position
// error of the FP32 local ray.  A leaf whose inflated box is hit is a
// candidate with entry bounds [lo, hi] (hi only if the deflated box is hit:
// "certain").  A ray is certified when the candidate with the smallest lo is
// certain, every other candidate's lo exceeds its hi, and its [lo, hi] is
// narrower than 2^-17 of its t; otherwise it is flagged and, with FP64_FIX,
// recomputed in FP64 by k_fix (whose arithmetic needs no certification).
//
// Traversal: children of a node are visited in the order their entry t
// increases.  With every direction component made non-negative by mirroring,
// the entry of child m is max(T0, max over axes in m of the mid-plane t), so
// the order follows from sorting the three mid-plane t values; a per-block
// table gives the first child of a mask in that order.  A stack holds, per
// level, the parent's descriptor, the children still to visit and their order.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdint>
#include <memory>
#include <mutex>
#include <type_traits>
#include <vector>

#include "svo_internal.h"

namespace svo {

template <int NI>
struct TraceLaunchT {
  TraceItem items[NI];
  int32_t n_items;
  uint32_t flags;
  unsigned long long n_tiles;
  unsigned long long *tile_counter;
  unsigned long long *fix_list;
  unsigned int *fix_count;
  unsigned long long fix_capacity;
  uint4 *fix_cand;                  // pool of stored leaves (winner, contenders or re-trace cap)
  unsigned long long cand_capacity; // pool entries
  unsigned int *cand_count;         // pool entries taken
  uint32_t *fix_off;                // per list slot: its first pool entry, or kNoCand
  svo_trace_stats *stats;
  unsigned int *err;
  int32_t same_scene;    // every item traces the same scene
  int32_t cull_chunk;    // tiles a block of the culling launch claims at a time
  int32_t one_scene;     // every item traces the same scene: stage its tables in shared memory
  int32_t stack_levels;  // traversal stack levels per thread (max asset depth - 1)
  int32_t mbox_words;    // grid walk: words of each thread's tested-part bitset (max parts / 32)
  int32_t block;         // threads per block of the trace kernel: 64, 128 or 256
  int32_t rays_per_lane; // rays per lane in a warp's tile (tile = 32 * rays_per_lane rays)
  const int2 *top;       // one_scene: per part (first, count) of its top-level nodes staged in shared memory
  int32_t top_nodes;     // staged nodes per block (0: none)
  int32_t top_levels;    // levels staged of every part
  QueueEntry *queue;                // SVO_TRACE_WAVEFRONT: the ray queue (item i from items[i].qbase)
  unsigned int *queue_count;        // SVO_TRACE_WAVEFRONT: entries queued per item
  unsigned long long *queue_tile;   // SVO_TRACE_WAVEFRONT: tile counter of the descent launch
  TileEntry *tiles;                 // tile-culled image trace: the tiles to trace
  unsigned int *tile_count;         // their number
  unsigned int *gate_count;         // see TraceLaunch
  unsigned int gate;
  unsigned long long *clean;        // the FP64 pass leaves these kCounterWords at zero, and every dirty flag (nullptr: no)
};

namespace {

constexpr float kU = 5.9604644775390625e-8f;   // 2^-24, FP32 unit roundoff
constexpr float kTau = 7.62939453125e-6f;      // 2^-17
constexpr int kCap = 4;  // candidate parts per pass (4: 1.5-2% faster than 8, fewer live registers)
constexpr int kSmemParts = 256;                 // parts staged in shared memory
constexpr int kBlock = 128;  // block size of the FP64 pass; the trace kernel takes 64, 128 or 256
// Resident threads per SM the trace kernel's register allocation must allow
// (768 = 24 warps: at most 80 registers a thread).  Measured at 24 / 20 / 16
// warps: 2.1 M incoherent rays against 128 parts 0.712 / 0.766 / 0.857 ms, a
// 1920x1080 frame of a 16-part figure 0.160 / 0.150 / 0.150 ms.  The counting
// (STATS) and hit-buffer (REUSE) builds keep 16 warps: they would spill more.
constexpr int kTraceThreadsPerSM = 768;
// The image-tile launch (LIST) keeps 16 warps: with the culling done before,
// it runs only tiles that descend (nine requests, 6.7 M rays: 0.707 ms, 0.691
// at 20 warps; 2.1 M rays against 1024 parts: 0.249 and 0.245).
constexpr int kListThreadsPerSM = 512;
// Image tiles in one launch keep 16 warps as well: their coherent lanes fill
// the issue slots, and 128 registers do without spills.  24 / 20 / 16 warps: a
// 1920x1080 frame of a 16-part figure 0.158 / 0.153 / 0.151 ms alone and 183 /
// 175 / 165 us a call with others behind it.
constexpr int kImageThreadsPerSM = 512;

constexpr unsigned long long kRayBits = 40;
constexpr uint32_t kNoCand = 0xFFFFFFFFu;  // a list slot without stored leaves

// Child masks of the descent: mirror[mir][mask] is a node's child mask with
// the octants mirrored along the axes in mir; first[p][mask] the first child
// of a (mirrored) mask in the order of their entries, p = (Bx <= By) |
// (Bx <= Bz) << 1 | (By <= Bz) << 2 for the mid-plane parameters B.
struct Tables {
  uint8_t mirror[8][256];
  uint8_t first[8][256];
};
constexpr size_t kTablesBytes = (sizeof(Tables) + 15) & ~size_t(15);

__device__ void build_tables(Tables *t) {
  for (int e = threadIdx.x; e < 8 * 256; e += blockDim.x) {
    const int a = e >> 8, mask = e & 255;
    uint32_t mirrored = 0, first = 0;
    // A child's entry is the largest B of its far axes, so the children come
    // in the order of the sums of 1 << rank over those axes, rank 0 for the
    // smallest B.
    const int xy = a & 1, xz = (a >> 1) & 1, yz = (a >> 2) & 1;
    const int rx = 2 - xy - xz, ry = 1 + xy - yz, rz = xz + yz;
    int best = 64;
    for (int m = 0; m < 8; ++m) {
      if ((mask >> m) & 1) mirrored |= 1u << (m ^ a);
      const int q = (m & 1 ? 1 << rx : 0) + (m & 2 ? 1 << ry : 0) + (m & 4 ? 1 << rz : 0);
      if (((mask >> m) & 1) && q < best) {
        best = q;
        first = (uint32_t)m;
      }
    }
    t->mirror[a][mask] = (uint8_t)mirrored;
    t->first[a][mask] = (uint8_t)first;
  }
}

// The tables are built once per device (svo_ctx_create) and copied into
// shared memory by every block.
__device__ __align__(16) Tables g_tables;

__global__ void k_init_tables() { build_tables(&g_tables); }

__device__ __forceinline__ void load_tables(Tables *t) {
  static_assert(sizeof(Tables) % 16 == 0, "Tables must be a whole number of 16-byte words");
  const uint4 *src = reinterpret_cast<const uint4 *>(&g_tables);
  uint4 *dst = reinterpret_cast<uint4 *>(t);
  for (int i = threadIdx.x; i < (int)(sizeof(Tables) / 16); i += blockDim.x) dst[i] = src[i];
}

template <typename R>
struct Num;
template <>
struct Num<float> {
  __device__ static float inf() { return __int_as_float(0x7f800000); }
};
template <>
struct Num<double> {
  __device__ static double inf() { return __longlong_as_double(0x7ff0000000000000ll); }
  __device__ static double pow2neg(int l) { return __longlong_as_double((long long)(1023 - l) << 52); }
};
constexpr float kTinyDir = 1e-30f;  // direction components are at least this along a descent
__device__ __forceinline__ float pow2neg(int l) { return __int_as_float((127 - l) << 23); }

// FP32 per-ray state of the certified closest-hit search.
struct CertState {
  float lo1, hi1, te1;  // candidate with the smallest (lo, part, voxel)
  float lo2;            // smallest lo of all other candidates
  float hi_min;         // smallest hi of the certain candidates (prune bound)
  uint32_t part1;
  uint32_t cert1;
  unsigned long long vox1;
};

// FP64 per-ray state of the exact closest-hit search.
struct ExactState {
  double t;
  uint32_t part;
  unsigned long long vox;
};

// A ray in a part's frame in FP64: the origin, and one reciprocal per axis
// instead of two divisions a leaf (the result differs from the quotient by at
// most an ulp or two); inv = 0 stands for a zero direction component.
struct LocalRay64 {
  double o[3], inv[3];
};

__device__ __forceinline__ LocalRay64 local_ray64(const double *__restrict__ m, float4 o, float4 d) {
  const double ox = o.x, oy = o.y, oz = o.z, dx = d.x, dy = d.y, dz = d.z;
  LocalRay64 l;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    l.o[k] = fma(m[4 * k], ox, fma(m[4 * k + 1], oy, fma(m[4 * k + 2], oz, m[4 * k + 3])));
    const double ld = fma(m[4 * k], dx, fma(m[4 * k + 1], dy, m[4 * k + 2] * dz));
    l.inv[k] = ld != 0.0 ? 1.0 / ld : 0.0;
  }
  return l;
}

// Closed-box entry of one leaf in FP64 (the definition the oracle follows):
// slab test of the leaf cell's box between tmin and tmax; a zero direction
// component keeps the slab only if the origin lies in it.  Returns whether
// the leaf is hit and its candidate t.  FP64 issues at two lanes per clock
// and SM, so its instructions are what this costs: the near plane is picked
// by the sign bit of the reciprocal, and the far corner is the near one plus
// a leaf (exact).
__device__ __forceinline__ bool leaf_entry64(const LocalRay64 &l, int D, unsigned long long vox, float tmin,
                                             float tmax, double &t) {
  const uint32_t mask = (1u << D) - 1u;
  const double s = Num<double>::pow2neg(D);
  double t0 = (double)tmin, t1 = (double)tmax;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double blo = (double)((uint32_t)(vox >> (k * D)) & mask) * s, bhi = blo + s;
    const long long bits = __double_as_longlong(l.inv[k]);
    if (bits == 0) {
      if (l.o[k] < blo || l.o[k] > bhi) return false;
      continue;
    }
    const double ta = (blo - l.o[k]) * l.inv[k], tb = (bhi - l.o[k]) * l.inv[k];
    const double near = bits < 0 ? tb : ta, far = bits < 0 ? ta : tb;
    t0 = near > t0 ? near : t0;
    t1 = far < t1 ? far : t1;
  }
  t = t0;
  return t0 <= t1;
}

// Leaves that may still be the closest hit: every candidate whose entry lower
// bound lo does not exceed hi_min (the best upper bound of a certainly hit
// leaf).  The true winner is always among them, so a flagged ray can be
// resolved by intersecting only these leaves in FP64.
struct Contenders {
  float lo[kContenders];
  uint32_t part[kContenders];
  unsigned long long vox[kContenders];
  int n;
  bool overflow;
};

__device__ __forceinline__ void keep_contender(Contenders &c, float hi_min, float lo, uint32_t part,
                                               unsigned long long vox) {
  if (!(lo <= hi_min)) return;
  if (c.n < kContenders) {
    c.lo[c.n] = lo;
    c.part[c.n] = part;
    c.vox[c.n] = vox;
    ++c.n;
    return;
  }
  for (int i = 0; i < kContenders; ++i) {
    if (!(c.lo[i] <= hi_min)) {  // no longer a contender: reuse its slot
      c.lo[i] = lo;
      c.part[i] = part;
      c.vox[i] = vox;
      return;
    }
  }
  c.overflow = true;
}

__device__ __forceinline__ void offer_state(CertState &s, float lo, float hi, float te, bool cert, uint32_t part,
                                            unsigned long long vox) {
  const bool better = lo < s.lo1 || (lo == s.lo1 && (part < s.part1 || (part == s.part1 && vox < s.vox1)));
  if (better) {
    s.lo2 = fminf(s.lo2, s.lo1);
    s.lo1 = lo;
    s.hi1 = hi;
    s.te1 = te;
    s.part1 = part;
    s.vox1 = vox;
    s.cert1 = cert ? 1u : 0u;
  } else {
    s.lo2 = fminf(s.lo2, lo);
  }
}

__device__ __forceinline__ void offer(CertState &s, Contenders &c, float lo, float hi, float te, bool cert,
                                      uint32_t part, unsigned long long vox) {
  if (cert) s.hi_min = fminf(s.hi_min, hi);
  keep_contender(c, s.hi_min, lo, part, vox);
  offer_state(s, lo, hi, te, cert, part, vox);
}

__device__ __forceinline__ void offer(ExactState &s, double t, uint32_t part, unsigned long long vox) {
  if (t < s.t || (t == s.t && (part < s.part || (part == s.part && vox < s.vox)))) {
    s.t = t;
    s.part = part;
    s.vox = vox;
  }
}

__device__ __forceinline__ float prune_bound(const CertState &s, float tmax) { return fminf(tmax, s.hi_min); }
// The same bound in a part's shifted parameter t_rel = t - tshift, rounded up
// so that pruning stays conservative.
__device__ __forceinline__ float rel_bound(const CertState &s, float tmax_rel, float tshift) {
  return fminf(tmax_rel, __fsub_ru(s.hi_min, tshift));
}

struct Counters {
  uint32_t parts_tested, parts_entered, nodes, leaves, passes;
  uint32_t f_winner, f_overlap, f_width, reused;
};

// Descriptor idx, a node of level `lev`, of a part.  The node array is
// breadth first, so the nodes of the top `top_levels` levels are its first
// ones; those come from the block's shared-memory copy at address `top`
// (32-bit shared address of the part's first staged node), the rest from
// global memory.
__device__ __forceinline__ uint2 node_at(const uint2 *__restrict__ nodes, uint32_t top, int top_levels, int lev,
                                         uint32_t idx) {
  if (top_levels > 0 && lev < top_levels) {  // folds away where top_levels is the constant 0
    uint2 v;
    asm("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(top + 8u * idx));
    return v;
  }
  return __ldg(&nodes[idx]);
}

// One part's front-to-back descent in progress: what the descent keeps
// between node visits (its stack lives in shared memory).  The local ray
// has every direction component made non-negative by mirroring (mir: the
// mirrored axes), with reciprocals (ix, iy, iz).
//
// Node corners are kept as floats in [1, 2): 1 + the corner.  Their mantissa
// bits are the path from the root, one per level and axis, so a step down
// sets a bit, a pop clears the bits below its level, and a plane needs no
// conversion from integers.  A plane P (so shifted) inflated by eta along the
// ray is crossed at P ix + lx (its lower side) or P ix + hx (its upper side),
// lx = -((o + 1) + eta) ix, hx = -((o + 1) - eta) ix, rounded outward: one FMA
// each.
struct Descent {
  float ix, iy, iz, lx, ly, lz, hx, hy, hz, ox, oy, oz, tmin, tmax, tshift;
  const uint2 *nodes;
  uint32_t n_nodes, part, top, mir;
  int D, top_levels, level;
  uint32_t X, Y, Z;  // the node's lower corner + 1, as float bits
  uint32_t live;     // bit l: the stack entry of level l still has a child that may hold the closest hit
  uint2 desc;        // the descriptor of the node visited next
};

// Starts a descent at the part's root (the caller has checked n_nodes > 0).
// (o, d): the local ray, whose parameter is t - tshift; tmin / tmax in that
// parameter.
template <bool STATS>
__device__ __forceinline__ void descent_start(Descent &s, const uint2 *__restrict__ nodes, uint32_t n_nodes,
                                              uint32_t top, int top_levels, int D, float ox, float oy, float oz,
                                              float dx, float dy, float dz, float tmin, float tmax, float eta,
                                              float tshift, uint32_t part, Counters &cnt) {
  // The planes' constants: the origin shifted by one (mirrored axis: o -> 1 - o,
  // so 2 - o), eta to either side, times 1/d, every step rounded outward (u up, d
  // down).  Holding corners in [1, 2) puts |1 + o| where |o| was, and rounded to
  // nearest these three roundings needed 6 |1 + o| units more of eta for every
  // plane; rounded outward they cost a plane what they are, half a unit each on
  // average.  60 K rays that graze or frame depth-13 parts: 28.5 K uncertain with
  // corners in [1, 2) and rounded to nearest, 27.9 K with corners in [0, 1), 27.6 K
  // now (depth 9: 11.9, 11.2, 10.9 K).
  uint32_t mir = 0;
  float ux = __fadd_ru(1.0f, ox), uy = __fadd_ru(1.0f, oy), uz = __fadd_ru(1.0f, oz);
  float lx = __fadd_rd(1.0f, ox), ly = __fadd_rd(1.0f, oy), lz = __fadd_rd(1.0f, oz);
  if (dx < 0.f) {
    ux = __fsub_ru(2.0f, ox);
    lx = __fsub_rd(2.0f, ox);
    ox = 1.0f - ox;
    dx = -dx;
    mir |= 1u;
  }
  if (dy < 0.f) {
    uy = __fsub_ru(2.0f, oy);
    ly = __fsub_rd(2.0f, oy);
    oy = 1.0f - oy;
    dy = -dy;
    mir |= 2u;
  }
  if (dz < 0.f) {
    uz = __fsub_ru(2.0f, oz);
    lz = __fsub_rd(2.0f, oz);
    oz = 1.0f - oz;
    dz = -dz;
    mir |= 4u;
  }
  s.ix = __frcp_rn(fmaxf(dx, kTinyDir));
  s.iy = __frcp_rn(fmaxf(dy, kTinyDir));
  s.iz = __frcp_rn(fmaxf(dz, kTinyDir));
  s.lx = -__fmul_ru(__fadd_ru(ux, eta), s.ix);
  s.ly = -__fmul_ru(__fadd_ru(uy, eta), s.iy);
  s.lz = -__fmul_ru(__fadd_ru(uz, eta), s.iz);
  s.hx = -__fmul_rd(__fsub_rd(lx, eta), s.ix);
  s.hy = -__fmul_rd(__fsub_rd(ly, eta), s.iy);
  s.hz = -__fmul_rd(__fsub_rd(lz, eta), s.iz);
  s.ox = ox;
  s.oy = oy;
  s.oz = oz;
  s.tmin = tmin;
  s.tmax = tmax;
  s.tshift = tshift;
  s.nodes = nodes;
  s.n_nodes = n_nodes;
  s.part = part;
  s.top = top;
  s.mir = mir;
  s.D = D;
  s.top_levels = top_levels;
  s.level = 0;
  s.X = s.Y = s.Z = 0x3F800000u;
  s.live = 0;
  s.desc = node_at(nodes, top, top_levels, 0, 0u);
  if (STATS) ++cnt.nodes;
}

// The planes of the node a descent is at: T0 its inflated entry (not before
// tmin), T1 its inflated exit, B and C the entry into the far and the exit
// from the near half along each axis, both inflated.
struct NodePlanes {
  float h, T0, T1, Bx, By, Bz, Cx, Cy, Cz;

  __device__ __forceinline__ explicit NodePlanes(const Descent &s) {
    const float sz = pow2neg(s.level);
    h = sz * 0.5f;
    const float px = __uint_as_float(s.X), py = __uint_as_float(s.Y), pz = __uint_as_float(s.Z);
    const float mx = px + h, my = py + h, mz = pz + h;
    T0 = fmaxf(fmaxf(fmaf(px, s.ix, s.lx), fmaf(py, s.iy, s.ly)), fmaxf(fmaf(pz, s.iz, s.lz), s.tmin));
    T1 = fminf(fminf(fmaf(px + sz, s.ix, s.hx), fmaf(py + sz, s.iy, s.hy)), fmaf(pz + sz, s.iz, s.hz));
    Bx = fmaf(mx, s.ix, s.lx);
    By = fmaf(my, s.iy, s.ly);
    Bz = fmaf(mz, s.iz, s.lz);
    Cx = fmaf(mx, s.ix, s.hx);
    Cy = fmaf(my, s.iy, s.hy);
    Cz = fmaf(mz, s.iz, s.hz);
  }

  // Mask of the children (mirrored octants m) whose inflated boxes the ray
  // meets up to tl: max(T0, B_i : i in m) <= min(T1, tl, C_j : j not in m).
  __device__ __forceinline__ uint32_t hits(float tl) const {
    constexpr uint32_t FX = 0xAAu, FY = 0xCCu, FZ = 0xF0u;  // children in the far half of each axis
    const float T = fminf(T1, tl);
    uint32_t hit = (T0 <= T) ? 0xFFu : 0u;
    hit &= (Bx <= T) ? 0xFFu : ~FX;
    hit &= (By <= T) ? 0xFFu : ~FY;
    hit &= (Bz <= T) ? 0xFFu : ~FZ;
    hit &= (Cx >= T0) ? 0xFFu : FX;
    hit &= (Cy >= T0) ? 0xFFu : FY;
    hit &= (Cz >= T0) ? 0xFFu : FZ;
    hit &= (Bx <= Cy) ? 0xFFu : ~(FX & ~FY);
    hit &= (Bx <= Cz) ? 0xFFu : ~(FX & ~FZ);
    hit &= (By <= Cx) ? 0xFFu : ~(FY & ~FX);
    hit &= (By <= Cz) ? 0xFFu : ~(FY & ~FZ);
    hit &= (Bz <= Cx) ? 0xFFu : ~(FZ & ~FX);
    hit &= (Bz <= Cy) ? 0xFFu : ~(FZ & ~FY);
    return hit;
  }

  // The row of Tables::first for the order of the three mid-planes.
  __device__ __forceinline__ uint32_t order() const {
    return (Bx <= By ? 1u : 0u) | (Bx <= Bz ? 2u : 0u) | (By <= Bz ? 4u : 0u);
  }

  // Entry of child m: max(T0, B_i : i in m).
  __device__ __forceinline__ float entry(uint32_t m) const {
    float lo = T0;
    if (m & 1u) lo = fmaxf(lo, Bx);
    if (m & 2u) lo = fmaxf(lo, By);
    if (m & 4u) lo = fmaxf(lo, Bz);
    return lo;
  }
};

// Voxel id of leaf child m of the level D-1 node a descent is at.
__device__ __forceinline__ unsigned long long leaf_voxel(const Descent &s, uint32_t m) {
  const int D = s.D;
  const uint32_t flip = (1u << D) - 1u;
  uint32_t vx = ((s.X & 0x7FFFFFu) >> (23 - D)) + (m & 1u);
  uint32_t vy = ((s.Y & 0x7FFFFFu) >> (23 - D)) + ((m >> 1) & 1u);
  uint32_t vz = ((s.Z & 0x7FFFFFu) >> (23 - D)) + (m >> 2);
  if (s.mir & 1u) vx ^= flip;
  if (s.mir & 2u) vy ^= flip;
  if (s.mir & 4u) vz ^= flip;
  return (unsigned long long)vx | ((unsigned long long)vy << D) | ((unsigned long long)vz << (2 * D));
}

// Leaf child m of a node: the entry dlo into its deflated box (certain: that
// box is met), and the entry te into the box itself.
struct LeafBounds {
  float dlo, te;
  bool cert;
  __device__ __forceinline__ LeafBounds(const Descent &s, float h, uint32_t m) {
    float px = __uint_as_float(s.X), py = __uint_as_float(s.Y), pz = __uint_as_float(s.Z);
    if (m & 1u) px += h;
    if (m & 2u) py += h;
    if (m & 4u) pz += h;
    dlo = fmaxf(fmaxf(fmaf(px, s.ix, s.hx), fmaf(py, s.iy, s.hy)), fmaxf(fmaf(pz, s.iz, s.hz), s.tmin));
    const float dhi = fminf(fminf(fmaf(px + h, s.ix, s.lx), fmaf(py + h, s.iy, s.ly)),
                            fminf(fmaf(pz + h, s.iz, s.lz), s.tmax));
    // the corner itself is exact: p lies in [1, 2)
    te = fmaxf(fmaxf(((px - 1.0f) - s.ox) * s.ix, ((py - 1.0f) - s.oy) * s.iy),
               fmaxf(((pz - 1.0f) - s.oz) * s.iz, s.tmin));
    cert = dlo <= dhi;
  }
};

// One node of a descent, the certified search in FP32 with boxes inflated by
// eta: leaves give entry bounds.
// The node's child mask comes first, then its leaves, or the stack entry of
// this node, or -- with nothing to visit here -- that of the deepest level
// above that still has a child to visit; the step to that child is the same
// for both, so the lanes that descend and those that pop take it together.
// Returns false once the part is done.
//
// Bound by instruction issue and latency: the lanes of a warp descend, test
// leaves and pop in the same iteration, so its length is the sum of the paths
// (about 300 instructions and 1.3 us with integer corners, twelve
// inflated planes, and a step of its own for pops), and a launch is as long
// as its slowest tile, the visits of whose longest ray (150) follow each
// other.  With the corners as floats, eta inside the planes and one step for
// both: 1920x1080 frame of a 16-part figure 0.196 -> 0.160 ms, 2.1 M
// incoherent rays 0.954 -> 0.712, 1.05 M rays into depth-13 parts 1.455 ->
// 0.973.
template <bool STATS, int STRIDE>
__device__ __forceinline__ bool descent_step(Descent &s, uint2 *__restrict__ stk, const Tables *__restrict__ tab,
                                             CertState &st, Contenders &con, unsigned int &err, Counters &cnt) {
  int level = s.level;
  uint2 e;     // .x first child, .y child mask | children to visit (mirrored) << 8 | order << 16
  uint32_t m;  // the child to step to
  bool alive = true;  // one exit: a return in between would leave the lanes apart until the part's end
  {
    const NodePlanes nd(s);
    uint32_t hit = nd.hits(rel_bound(st, s.tmax, s.tshift)) & tab->mirror[s.mir][s.desc.y & 0xFFu];
    const uint32_t p = nd.order();
    if (hit != 0u && level == s.D - 1) {
      // children are leaves: test them in visiting order
      do {
        m = tab->first[p][hit];
        hit &= ~(1u << m);
        const float lo = nd.entry(m);
        if (lo > rel_bound(st, s.tmax, s.tshift)) break;  // later leaves start even later
        if (STATS) ++cnt.leaves;
        const unsigned long long vox = leaf_voxel(s, m);
        const LeafBounds lb(s, nd.h, m);
        // back to the ray's own parameter, rounding the bounds outward
        offer(st, con, __fadd_rd(s.tshift, lo), lb.cert ? __fadd_ru(s.tshift, lb.dlo) : Num<float>::inf(),
              s.tshift + lb.te, lb.cert, s.part, vox);
      } while (hit != 0u);
      hit = 0u;
    }
    e = make_uint2(s.desc.x, s.desc.y | (hit << 8) | (p << 16));  // above the leaves a node's leaf mask is 0
    m = tab->first[p][hit];
    if (hit == 0u) {
      // pop to the deepest level above that still has a child to visit
      uint32_t cand = s.live & ((1u << level) - 1u);
      bool found = false;
      while (cand != 0u && !found) {
        level = 31 - __clz(cand);
        const uint32_t keep = ~0u << (23 - level);
        s.X &= keep;
        s.Y &= keep;
        s.Z &= keep;
        e = stk[level * STRIDE];
        m = tab->first[e.y >> 16][(e.y >> 8) & 0xFFu];
        // the child's entry, but for its parent's; past the bound, it and all
        // later siblings are too far for good (the bound only shrinks)
        const float h = pow2neg(level + 1);
        float en = -Num<float>::inf();
        if (m & 1u) en = fmaf(__uint_as_float(s.X) + h, s.ix, s.lx);
        if (m & 2u) en = fmaxf(en, fmaf(__uint_as_float(s.Y) + h, s.iy, s.ly));
        if (m & 4u) en = fmaxf(en, fmaf(__uint_as_float(s.Z) + h, s.iz, s.lz));
        found = !(en > rel_bound(st, s.tmax, s.tshift));
        cand &= ~(1u << level);
      }
      s.live = found ? cand | (1u << level) : 0u;
      alive = found;
    }
  }
  // to child m of the node of `level` that e describes
  if (alive) {
    const uint32_t rest = e.y & ~(0x100u << m);
    const uint32_t bit = 1u << level;
    s.live &= ~bit;
    if (rest & 0xFF00u) {
      s.live |= bit;
      stk[level * STRIDE] = make_uint2(e.x, rest);
    }
    const uint32_t k = m ^ s.mir;
    const uint32_t idx = e.x + __popc(e.y & ((1u << k) - 1u));
    const uint32_t half = 1u << (22 - level);
    s.X += (m & 1u) * half;
    s.Y += ((m >> 1) & 1u) * half;
    s.Z += (m >> 2) * half;
    s.level = level + 1;
    alive = idx < s.n_nodes;
    if (alive) s.desc = node_at(s.nodes, s.top, s.top_levels, level + 1, idx);
    if (!alive) err |= kErrNodeIndex;
    if (STATS && alive) ++cnt.nodes;
  }
  return alive;
}

struct RayW {
  float ox, oy, oz, tmin, dx, dy, dz, tmax;
  float inv_dd;
  float inv_len;  // 1/|d|
  float onorm;    // ||o||_inf
};

// Conservative ray / sphere test: sphere (c, R) is hit by the segment.  Eq. 4
// with a direction of any length: l = c - o, tc = (l.d)/|d|^2, the squared
// distance of the centre to the line is |l - tc d|^2.  Every rounding is
// spelled out: a part's entry is the reference of its descent, so the launch
// shapes agree bit for bit only if no compilation contracts it differently.
__device__ __forceinline__ bool sphere_test(const RayW &r, float lx, float ly, float lz, float R, float &tin,
                                            float &tc) {
  tc = __fmul_rn(fmaf(lz, r.dz, fmaf(ly, r.dy, __fmul_rn(lx, r.dx))), r.inv_dd);
  const float qx = fmaf(-tc, r.dx, lx), qy = fmaf(-tc, r.dy, ly), qz = fmaf(-tc, r.dz, lz);
  const float p2 = fmaf(qz, qz, fmaf(qy, qy, __fmul_rn(qx, qx)));
  const float R2 = __fmul_rn(R, R);
  if (!(p2 <= R2)) return false;
  const float half = sqrtf(__fmul_rn(__fsub_rn(R2, p2), r.inv_dd));
  const float tout = __fadd_rn(tc, half);
  tin = __fsub_rn(tc, half);
  return tout >= r.tmin && tin <= r.tmax;
}

// Part test.  The part's cube lies in its exact bounding sphere, so a ray that
// truly meets the cube passes once the FP32 test's own rounding is covered
// (16 u (|l|_1 + r) of slack).  tref: the reference parameter for the part's
// descent -- the sphere entry (or the closest approach on a miss), not before
// tmin.
__device__ __forceinline__ bool sphere_cull(const RayW &r, float4 s, float &tin, float &tref) {
  if (s.w < 0.f) return false;
  const float lx = s.x - r.ox, ly = s.y - r.oy, lz = s.z - r.oz;
  const float ln = __fadd_rn(__fadd_rn(fabsf(lx), fabsf(ly)), fabsf(lz));
  const float Rt = fmaf(16.0f * kU, __fadd_rn(ln, s.w), __fmul_rn(s.w, 1.0f + 9.5367431640625e-7f));
  float tc;
  const bool hit = sphere_test(r, lx, ly, lz, Rt, tin, tc);
  tref = fmaxf(hit ? tin : tc, r.tmin);
  return hit;
}

__device__ __forceinline__ bool part_cull(const RayW &r, const PartHot &ph, float &tin, float &tref) {
  return sphere_cull(r, ph.sphere, tin, tref);
}

__device__ __forceinline__ bool cluster_cull(const RayW &r, const Cluster &c) {
  const float4 s = c.sphere;
  if (s.w < 0.f) return false;
  const float lx = s.x - r.ox, ly = s.y - r.oy, lz = s.z - r.oz;
  const float ln = fabsf(lx) + fabsf(ly) + fabsf(lz);
  // covers every member test's slack 16 u (|l_m|_1 + r_m), |l_m|_1 <= |l|_1 + sqrt(3) R
  const float Rt = s.w * (1.0f + 9.5367431640625e-7f) + 48.0f * kU * (2.0f * ln + 3.8f * s.w);
  float tin, tc;
  return sphere_test(r, lx, ly, lz, Rt, tin, tc);
}

// Ray -> part frame (Eq. 3) and descent.  The origin is first moved along the
// ray to q = o + tref d (tref: sphere entry), and q is mapped relative to the
// sphere centre c, o' = Ainv (q - c) + c', with c' the FP64-accurate local
// coordinates of c: all FP32 arithmetic then works on numbers of order one.
// The descent's parameter is t - tref.  eta bounds the position error of the
// FP32 local ray over the part (in local units), doubled for safety:
//   q rounding            u ||Ainv||_inf ||q||_inf
//   q - c and Ainv (q-c)   5u ||Ainv||_inf ||q - c||_inf, c' rounding u |c'|
//   slabs                 2u (1 + |o'|): 1/d and the FMA, each relative to a plane's distance from the
//                         origin, at most 1 + |o'| (the planes' constants are rounded outward)
//   FP32 direction        4u ||Ainv||_inf (|c - q|_1 + r)
// stop: shared-memory address of the block's staged top-level nodes, of
// which each part has its top `top_levels` levels (pa.spare0 carries, as
// bits, the part's first staged node; 0 levels when nothing is staged).
// part_start sets up the descent (returns false when the part's box is
// missed, starts beyond the bound, or the part is empty); trace_part_f32
// runs it to the end.
template <bool STATS, typename S>
__device__ __forceinline__ bool part_start(const RayW &r, const PartHot &ph, const PartAux &pa, float tref,
                                           uint32_t part, uint32_t stop, int top_levels, const S &st,
                                           Descent &ds, Counters &cnt) {
  const float4 a = ph.r0, b = ph.r1, c = ph.r2;
  const float4 s = ph.sphere;
  const float qx = fmaf(tref, r.dx, r.ox), qy = fmaf(tref, r.dy, r.oy), qz = fmaf(tref, r.dz, r.oz);
  const float vx = qx - s.x, vy = qy - s.y, vz = qz - s.z;
  const float ox = fmaf(a.x, vx, fmaf(a.y, vy, fmaf(a.z, vz, a.w)));
  const float oy = fmaf(b.x, vx, fmaf(b.y, vy, fmaf(b.z, vz, b.w)));
  const float oz = fmaf(c.x, vx, fmaf(c.y, vy, fmaf(c.z, vz, c.w)));
  const float dx = fmaf(a.x, r.dx, fmaf(a.y, r.dy, a.z * r.dz));
  const float dy = fmaf(b.x, r.dx, fmaf(b.y, r.dy, b.z * r.dz));
  const float dz = fmaf(c.x, r.dx, fmaf(c.y, r.dy, c.z * r.dz));
  const float qn = fmaxf(fmaxf(fabsf(qx), fabsf(qy)), fabsf(qz));
  const float vn = fmaxf(fmaxf(fabsf(vx), fabsf(vy)), fabsf(vz));
  const float v1 = fabsf(vx) + fabsf(vy) + fabsf(vz);
  const float on = fmaxf(fmaxf(fabsf(ox), fabsf(oy)), fabsf(oz));
  const float cn = fmaxf(fmaxf(fabsf(a.w), fabsf(b.w)), fabsf(c.w));
  const float eta =
      kU * (2.0f * pa.n_ainv * (qn + 5.0f * vn + 4.0f * (v1 + fabsf(s.w))) + 2.0f * cn + 4.0f * on + 4.0f) * 1.001f;
  float tmin_rel = __fsub_rd(r.tmin, tref), tmax_rel = __fsub_ru(r.tmax, tref);
  // Clip the segment to the part's occupied box, inflated by 2 eta: one eta
  // for the local ray's error, one for this slab arithmetic (at most (4 + 3 |o'|)
  // u: the plane, the difference, 1/d and the product).  Every leaf lies in the
  // box, so no leaf the ray meets is entered before the clipped start or left
  // after the clipped end: no candidate is lost, the nodes outside the box along
  // the ray are never visited, and a part whose box the ray misses is not
  // descended at all.
  {
    const float o3[3] = {ox, oy, oz}, d3[3] = {dx, dy, dz};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float lo = pa.box_lo[k] - 2.0f * eta, hi = pa.box_hi[k] + 2.0f * eta;
      if (d3[k] == 0.f) {
        if (o3[k] < lo || o3[k] > hi) tmax_rel = -Num<float>::inf();
        continue;
      }
      const float inv = 1.0f / d3[k];
      float ta = (lo - o3[k]) * inv, tb = (hi - o3[k]) * inv;
      if (ta > tb) {
        const float x = ta;
        ta = tb;
        tb = x;
      }
      tmin_rel = fmaxf(tmin_rel, ta);
      tmax_rel = fminf(tmax_rel, tb);
    }
  }
  // nothing to do either when the box starts beyond the best certain hit so
  // far (the descent's own bound)
  if (!(tmin_rel <= tmax_rel) || tmin_rel > rel_bound(st, tmax_rel, tref)) return false;
  if (STATS) ++cnt.parts_entered;
  if (pa.n_nodes == 0) return false;
  descent_start<STATS>(ds, pa.nodes, pa.n_nodes, stop + 8u * __float_as_uint(pa.spare0), top_levels, pa.depth,
                              ox, oy, oz, dx, dy, dz, tmin_rel, tmax_rel, eta, tref, part, cnt);
  return true;
}

template <bool STATS, int STRIDE>
__device__ __forceinline__ void trace_part_f32(const RayW &r, const PartHot &ph, const PartAux &pa, float tref,
                                               uint32_t part, const Tables *tab, uint32_t stop, int top_levels,
                                               uint2 *stk, CertState &st, Contenders &con, unsigned int &err,
                                               Counters &cnt) {
  Descent ds;
  if (part_start<STATS, CertState>(r, ph, pa, tref, part, stop, top_levels, st, ds, cnt))
    while (descent_step<STATS, STRIDE>(ds, stk, tab, st, con, err, cnt)) {
    }
}

// Insert (t, p) into the sorted register list (ct, cp); the displaced largest
// entry is returned in (t, p).
__device__ __forceinline__ void list_insert(float (&ct)[kCap], float (&ce)[kCap], int (&cp)[kCap], float &t,
                                            float &e, int &p) {
#pragma unroll
  for (int i = 0; i < kCap; ++i) {
    const bool sw = t < ct[i] || (t == ct[i] && p < cp[i]);
    const float t2 = sw ? ct[i] : t, e2 = sw ? ce[i] : e;
    const int p2 = sw ? cp[i] : p;
    ct[i] = sw ? t : ct[i];
    ce[i] = sw ? e : ce[i];
    cp[i] = sw ? p : cp[i];
    t = t2;
    e = e2;
    p = p2;
  }
}

// Whether a grid may be walked: once it is ready, what its build wrote is
// visible to the caller, and it stays as it is until the scene's next refit.
__device__ __forceinline__ bool grid_ready(const SceneGrid *g) {
  int state;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(state) : "l"(&g->stale) : "memory");
  return state == kGridReady;
}

// Where a ray enters the scene grid: its first cell (cur), the step along
// each axis, 1/d (rd), the crossing of the cell's far plane per axis (tn) and
// the end of its segment in the grid's box (t1).  Returns whether it walks;
// ok: false for a ray the walk's arithmetic cannot take safely.
__device__ __forceinline__ bool grid_enter(const RayW &r, const SceneGrid &g, int (&cur)[3], int (&step)[3],
                                           float (&rd)[3], float (&tn)[3], float &t1, bool &ok) {
  const int G = g.G;
  const float o[3] = {r.ox, r.oy, r.oz}, d[3] = {r.dx, r.dy, r.dz};
  ok = true;
  // the segment inside the grid box
  float t0 = r.tmin;
  t1 = r.tmax;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float blo = g.lo[a], bhi = fmaf((float)G, g.cs[a], g.lo[a]);
    if (d[a] == 0.f) {
      if (o[a] < blo || o[a] > bhi) t1 = -Num<float>::inf();
      continue;
    }
    float ta = (blo - o[a]) / d[a], tb = (bhi - o[a]) / d[a];
    // else a component too small for the walk's arithmetic (the crossings
    // below stay within a few roundings of these, so they stay finite)
    ok = ok && fabsf(ta) < 1e38f && fabsf(tb) < 1e38f;
    if (ta > tb) {
      const float x = ta;
      ta = tb;
      tb = x;
    }
    t0 = fmaxf(t0, ta);
    t1 = fminf(t1, tb);
  }
  // the rounding allowance: a few units of roundoff of the largest magnitudes
  // in the crossing and start-cell arithmetic, against m/2 = 2^-11 cells
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float mag = fabsf(o[a]) + fabsf(g.lo[a]) + (float)G * g.cs[a] + fabsf(t0 * d[a]);
    ok = ok && 8.0f * kU * mag <= g.cs[a] * 4.8828125e-4f;
    const float f = (fmaf(t0, d[a], o[a]) - g.lo[a]) * g.inv_cs[a];
    const int i = (int)floorf(fminf(fmaxf(f, 0.f), (float)G));
    cur[a] = i > G - 1 ? G - 1 : i;
    step[a] = d[a] > 0.f ? 1 : (d[a] < 0.f ? -1 : 0);
    rd[a] = d[a] != 0.f ? 1.0f / d[a] : 0.f;
    tn[a] = d[a] != 0.f ? (fmaf((float)(cur[a] + (step[a] > 0 ? 1 : 0)), g.cs[a], g.lo[a]) - o[a]) * rd[a]
                        : Num<float>::inf();
  }
  return ok && t0 <= t1;  // t0 > t1: the segment misses every sphere box
}

// Culling through the scene-level grid (Sec. V-E).  Each cell lists every
// part whose sphere box comes within m = 2^-10 cells of it.  The ray walks the
// cells it crosses front to back (a 3D DDA whose crossing parameters are
// computed afresh from each cell plane, (plane - o) * (1/d), three roundings
// each, increasing along the walk); for t in the parameter interval of a visited cell
// the exact ray point lies within the rounding error of that cell, and a ray
// is only walked when that error is below m/2 (else the function returns
// false for it and the ray takes the cluster level).  The intervals of the
// visited cells follow each other without gaps, so a part whose sphere the
// exact ray meets at some t in them is listed in a visited cell.  Each listed
// part is sphere-tested once (a bitset per thread); the walk ends after the
// first cell whose interval reaches past the bound, the segment or the box.
//
// Called by the whole warp (go: this lane's ray takes part).  Each round,
// every walking lane gathers up to kCap candidates from its cell's list, and
// then the lanes descend their candidates together, in order of entry, so
// that the warp runs the descents side by side as on the cluster level.
template <bool STATS, int BLOCK>
__device__ __forceinline__ bool grid_walk(const RayW &r, bool go, const SceneGrid &g, const int32_t *cstart,
                                          const int32_t *cparts,
                                          const PartHot *__restrict__ hot, const PartAux *__restrict__ aux,
                                          const Tables *tab, uint32_t stop, int top_levels, uint2 *stk, uint32_t *mbox,
                                          int mwords, CertState &st, Contenders &con, unsigned int &err,
                                          Counters &cnt) {
  const int G = g.G;
  const float o[3] = {r.ox, r.oy, r.oz};
  int cur[3], step[3];
  float rd[3], tn[3], t1;
  bool ok;
  bool walking = grid_enter(r, g, cur, step, rd, tn, t1, ok) && go;
  int k = 0, kend = 0;
  if (walking) {
    for (int w = 0; w < mwords; ++w) mbox[w * BLOCK] = 0u;
    const int c = cur[0] + G * (cur[1] + G * cur[2]);
    k = cstart[c];
    kend = cstart[c + 1];
  }
  while (__any_sync(0xffffffffu, walking)) {
    float ct[kCap], ce[kCap];
    int cp[kCap];
#pragma unroll
    for (int i = 0; i < kCap; ++i) {
      ct[i] = Num<float>::inf();
      ce[i] = 0.f;
      cp[i] = 0x7fffffff;
    }
    if (walking) {
      // gather: the next candidates of this cell, up to kCap
      int n = 0;
      while (k < kend && n < kCap) {
        const int p = cparts[k++];
        uint32_t *wp = mbox + (p >> 5) * BLOCK;
        const uint32_t bit = 1u << (p & 31), wv = *wp;
        if (wv & bit) continue;
        *wp = wv | bit;
        float tin, tref;
        if (STATS) ++cnt.parts_tested;
        if (!part_cull(r, hot[p], tin, tref)) continue;
        if (tin > prune_bound(st, r.tmax)) continue;  // the bound only shrinks: never needed
        int pp = p;
        list_insert(ct, ce, cp, tin, tref, pp);  // not full: nothing is pushed out
        ++n;
      }
    }
    // descend, the warp's lanes side by side (the list shifts down each step)
#pragma unroll 1
    for (int i = 0; i < kCap && __any_sync(0xffffffffu, ct[0] != Num<float>::inf()); ++i) {
      if (ct[0] != Num<float>::inf() && ct[0] <= prune_bound(st, r.tmax))
        trace_part_f32<STATS, BLOCK>(r, hot[cp[0]], aux[cp[0]], ce[0], (uint32_t)cp[0], tab, stop,
                                                top_levels, stk, st, con, err, cnt);
#pragma unroll
      for (int j = 0; j < kCap - 1; ++j) {
        ct[j] = ct[j + 1];
        ce[j] = ce[j + 1];
        cp[j] = cp[j + 1];
      }
      ct[kCap - 1] = Num<float>::inf();
    }
    if (walking && k >= kend) {
      // the cell's exit: the nearest crossing of a far cell plane
      const int ax = tn[0] <= tn[1] ? (tn[0] <= tn[2] ? 0 : 2) : (tn[1] <= tn[2] ? 1 : 2);
      const float tx = fminf(fminf(tn[0], tn[1]), tn[2]);
      if (!(tx < t1) || tx > prune_bound(st, r.tmax)) {  // also: no axis moves (tx infinite)
        walking = false;
      } else {
        bool out = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {  // static indices keep the arrays in registers
          if (a != ax) continue;
          cur[a] += step[a];
          out = cur[a] < 0 || cur[a] > G - 1;
          tn[a] = (fmaf((float)(cur[a] + (step[a] > 0 ? 1 : 0)), g.cs[a], g.lo[a]) - o[a]) * rd[a];
        }
        if (out) {
          walking = false;
        } else {
          const int c = cur[0] + G * (cur[1] + G * cur[2]);
          k = cstart[c];
          kend = cstart[c + 1];
        }
      }
    }
  }
  return ok;
}

// One culling pass (Sec. IV-A/B): the ray against the cluster spheres, then
// against the part spheres of the clusters it meets; the first kCap
// candidates in order of sphere entry (entry t, descent reference parameter,
// part) that come after (last_t, last_p), the last part an earlier pass
// descended, and in over_t the smallest entry that did not fit the list.
// Called by the whole warp (need: this lane's ray takes part); NC must be
// the same on every lane.  Every lane that met a cluster tests all its
// members; with VOTE the others idle through them, and a cluster no lane
// met is skipped.  VOTE false: a lane alone (no warp vote; its warp's lanes
// may hold rays of different items), as the refilling descent launch calls
// it.
template <bool STATS, bool VOTE = true>
__device__ __forceinline__ void cull_pass(const RayW &r, bool need, int NC, const PartHot *__restrict__ hot,
                                          const Cluster *__restrict__ cl, const int32_t *__restrict__ order,
                                          float last_t, int last_p, float (&ct)[kCap], float (&ce)[kCap],
                                          int (&cp)[kCap], float &over_t, Counters &cnt) {
  for (int c = 0; c < NC; ++c) {
    const Cluster cc = cl[c];
    const bool hc = need && cluster_cull(r, cc);
    if (VOTE && __ballot_sync(0xffffffffu, hc) == 0u) continue;  // no lane needs this cluster
    if (hc) {
      const uint32_t fc = __float_as_uint(cc.aux.w);
      const int first = (int)(fc & 0xFFFFu), count = (int)(fc >> 16);
      for (int k = 0; k < count; ++k) {
        const int p = order[first + k];
        float tin, eta;
        if (STATS) ++cnt.parts_tested;
        if (!part_cull(r, hot[p], tin, eta)) continue;
        if (tin < last_t || (tin == last_t && p <= last_p)) continue;  // visited in an earlier pass
        float t = tin, e = eta;
        int pp = p;
        list_insert(ct, ce, cp, t, e, pp);
        over_t = fminf(over_t, t);
      }
    }
  }
}

// The first culling pass of the culling launch through the scene grid, one
// ray a lane and resumable: the parts listed in the cells the ray crosses are
// tested as it walks on (the walk and its guarantee are grid_walk's).  Every
// part whose sphere the exact ray meets is listed in some visited cell, so
// the candidates are those of the cluster level but for parts the ray misses
// by the tests' slack, which hold no leaf it meets.  A part listed in several
// cells is tested in each: the grids this is used for list about one part a
// cell, so that costs less than a bitset, and only a part that is hit is
// looked up in the candidate list.
struct GridCull {
  float tn[3], rd[3], far_i[3], t1;  // crossings of the cell's far planes, 1/d, the planes' indices, the end
  int left[3];                       // cells left along each axis
  int c, k, end;                     // the cell, its next entry and its last
};

// cstart and cparts are the block's shared-memory copies of the grid's lists:
// 32 lanes in 32 cells read 32 different lines, which L1 serves one after
// another.  Returns whether the ray walks; ok: false for a ray the walk
// cannot take.
__device__ __forceinline__ bool grid_cull_start(const RayW &r, const SceneGrid &g, const uint16_t *cstart,
                                                GridCull &w, bool &ok) {
  int cur[3], step[3];
  if (!grid_enter(r, g, cur, step, w.rd, w.tn, w.t1, ok)) return false;
  const int G = g.G;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    w.far_i[a] = (float)(cur[a] + (step[a] > 0 ? 1 : 0));
    w.left[a] = step[a] > 0 ? G - 1 - cur[a] : cur[a];
  }
  w.c = cur[0] + G * (cur[1] + G * cur[2]);
  w.k = cstart[w.c];
  w.end = cstart[w.c + 1];
  return true;
}

// One part and -- once the cell's last is done -- one cell.  Returns false at
// the walk's end.  dims: the grid's corner and cell size per axis, G and G^2.
struct GridDims {
  float lo[3], cs[3];
  int stride[3];
};

__device__ __forceinline__ bool grid_cull_step(const RayW &r, const GridDims &g, const uint16_t *cstart,
                                               const uint16_t *cparts, const float4 *sphere, GridCull &w,
                                               float (&ct)[kCap], float (&ce)[kCap], int (&cp)[kCap],
                                               float &over_t) {
  if (w.k < w.end) {
    const int p = cparts[w.k++];
    float tin, tref;
    if (sphere_cull(r, sphere[p], tin, tref)) {
      bool seen = false;
#pragma unroll
      for (int i = 0; i < kCap; ++i) seen = seen || cp[i] == p;
      if (!seen) {
        int pp = p;
        list_insert(ct, ce, cp, tin, tref, pp);
        over_t = fminf(over_t, tin);
      }
    }
  }
  bool on = true;
  if (w.k >= w.end) {
    // the nearest crossing of a far cell plane
    const float tx = fminf(fminf(w.tn[0], w.tn[1]), w.tn[2]);
    const int ax = w.tn[0] <= w.tn[1] ? (w.tn[0] <= w.tn[2] ? 0 : 2) : (w.tn[1] <= w.tn[2] ? 1 : 2);
    const float o[3] = {r.ox, r.oy, r.oz};
    on = tx < w.t1;  // false also when no axis moves (tx infinite)
#pragma unroll
    for (int a = 0; a < 3; ++a) {  // static indices keep the arrays in registers
      if (a != ax) continue;
      on = on && w.left[a] != 0;
      --w.left[a];
      const bool up = w.rd[a] > 0.f;
      w.c += up ? g.stride[a] : -g.stride[a];
      w.far_i[a] += up ? 1.0f : -1.0f;
      w.tn[a] = (fmaf(w.far_i[a], g.cs[a], g.lo[a]) - o[a]) * w.rd[a];
    }
    if (on) {
      w.k = cstart[w.c];
      w.end = cstart[w.c + 1];
    }
  }
  return on;
}

// The first culling pass of the culling launch (the same candidates as
// cull_pass with nothing descended before), with the member tests packed
// over the warp's lanes across clusters.  Incoherent rays meet a cluster a
// few lanes at a time, and testing its members in place would leave most
// lanes idle.  So every (lane, cluster) pair of a cluster met by at most
// kInPlaceLanes lanes goes into the warp's ring in shared memory (owner
// lane, first | count << 16). Whenever four pairs wait, one round tests
// their 32 (pair, member) combinations: lane q takes member q & 7 of pair
// q >> 3 against its owner's ray (read by shuffles), and every hit goes back
// to the owner's list.  A cluster met by more lanes has its members tested
// in place.  The list keeps the kCap smallest (t, part) keys, and over_t the
// smallest t of the others, whatever the order of insertion, so the result
// is that of cull_pass.
constexpr int kPackRing = 64;      // ring slots per warp: a power of two above 3 + kInPlaceLanes
constexpr int kInPlaceLanes = 16;  // lanes above which a cluster's members are tested in place
static_assert(kClusterSize == 8 && kInPlaceLanes + 3 < kPackRing, "four pairs of eight members fill a round");

// One round: pairs ring[head .. head + n_pairs) (n_pairs <= 4), member
// lane & 7 of pair lane >> 3 on every lane.
template <bool STATS>
__device__ __forceinline__ void member_round(const RayW &r, const int2 *ring, int head, int n_pairs,
                                             const float4 *__restrict__ sph, const int32_t *__restrict__ order,
                                             float (&ct)[kCap], float (&ce)[kCap], int (&cp)[kCap],
                                             float &over_t, Counters &cnt) {
  const int lane = threadIdx.x & 31;
  const int e = lane >> 3, k = lane & 7;
  int owner = lane;
  uint32_t fc = 0u;  // no pair: count 0
  if (e < n_pairs) {
    const int2 q = ring[(head + e) & (kPackRing - 1)];
    owner = q.x;
    fc = (uint32_t)q.y;
  }
  const bool valid = k < (int)(fc >> 16);
  RayW ro;
  ro.ox = __shfl_sync(0xffffffffu, r.ox, owner);
  ro.oy = __shfl_sync(0xffffffffu, r.oy, owner);
  ro.oz = __shfl_sync(0xffffffffu, r.oz, owner);
  ro.dx = __shfl_sync(0xffffffffu, r.dx, owner);
  ro.dy = __shfl_sync(0xffffffffu, r.dy, owner);
  ro.dz = __shfl_sync(0xffffffffu, r.dz, owner);
  ro.tmin = __shfl_sync(0xffffffffu, r.tmin, owner);
  ro.tmax = __shfl_sync(0xffffffffu, r.tmax, owner);
  ro.inv_dd = __shfl_sync(0xffffffffu, r.inv_dd, owner);
  ro.inv_len = 0.f;
  ro.onorm = 0.f;
  float tin = 0.f, tref = 0.f;
  int p = 0;
  bool hit = false;
  if (valid) {
    const int q = (int)(fc & 0xFFFFu) + k;
    if (STATS) ++cnt.parts_tested;
    hit = sphere_cull(ro, sph[q], tin, tref);
    if (hit) p = order[q];
  }
  // hand each hit to its ray's lane (hits are rare: one round each)
  for (unsigned int hm = __ballot_sync(0xffffffffu, hit); hm != 0u; hm &= hm - 1u) {
    const int src = __ffs(hm) - 1;
    const int o = __shfl_sync(0xffffffffu, owner, src);
    float t = __shfl_sync(0xffffffffu, tin, src), te = __shfl_sync(0xffffffffu, tref, src);
    int pp = __shfl_sync(0xffffffffu, p, src);
    if (lane == o) {
      list_insert(ct, ce, cp, t, te, pp);
      over_t = fminf(over_t, t);
    }
  }
}

// ring: the warp's kPackRing slots.  Called by the whole warp.
template <bool STATS>
__device__ __forceinline__ void cull_first_packed(const RayW &r, bool need, int NC, const float4 *__restrict__ sph,
                                                  const Cluster *__restrict__ cl,
                                                  const int32_t *__restrict__ order, int2 *ring, float (&ct)[kCap],
                                                  float (&ce)[kCap], int (&cp)[kCap], float &over_t,
                                                  Counters &cnt) {
  const int lane = threadIdx.x & 31;
  int head = 0, pending = 0;  // warp-uniform: the ring's first waiting pair and the number waiting
  for (int c = 0; c < NC; ++c) {
    const Cluster cc = cl[c];
    const bool hc = need && cluster_cull(r, cc);
    const unsigned int m = __ballot_sync(0xffffffffu, hc);
    if (m == 0u) continue;  // no lane needs this cluster
    const uint32_t fc = __float_as_uint(cc.aux.w);
    const int nl = __popc(m);
    if (nl > kInPlaceLanes) {
      if (hc) {
        const int first = (int)(fc & 0xFFFFu), count = (int)(fc >> 16);
        for (int k = 0; k < count; ++k) {
          float tin, eta;
          if (STATS) ++cnt.parts_tested;
          if (!sphere_cull(r, sph[first + k], tin, eta)) continue;
          float t = tin, e = eta;
          int pp = order[first + k];
          list_insert(ct, ce, cp, t, e, pp);
          over_t = fminf(over_t, t);
        }
      }
      continue;
    }
    __syncwarp();  // the last round's reads of the ring are done
    if (hc) ring[(head + pending + __popc(m & ((1u << lane) - 1u))) & (kPackRing - 1)] = make_int2(lane, (int)fc);
    __syncwarp();
    pending += nl;
    for (; pending >= 4; pending -= 4, head = (head + 4) & (kPackRing - 1))
      member_round<STATS>(r, ring, head, 4, sph, order, ct, ce, cp, over_t, cnt);
  }
  for (; pending > 0; pending -= 4, head = (head + 4) & (kPackRing - 1))  // the last pairs
    member_round<STATS>(r, ring, head, min(pending, 4), sph, order, ct, ce, cp, over_t, cnt);
}

// cull_pass over the parts an image tile lists (k_tile_cull) in place of the
// clusters: the list holds every part whose part_cull any ray of the tile
// passes, so the candidates are those of cull_pass.  words: lane i holds
// word i & 15 of the tile's entry.  Called by the whole warp.
__device__ __forceinline__ void cull_listed(const RayW &r, bool need, uint32_t words, uint32_t count,
                                            const PartHot *__restrict__ hot, float last_t, int last_p,
                                            float (&ct)[kCap], float (&ce)[kCap], int (&cp)[kCap], float &over_t) {
  for (uint32_t k = 0; k < count; ++k) {
    const uint32_t w = __shfl_sync(0xffffffffu, words, 2 + (int)(k >> 1));
    const int p = (int)((w >> (16 * (k & 1u))) & 0xFFFFu);
    float tin, tref;
    if (!need || !part_cull(r, hot[p], tin, tref)) continue;
    if (tin < last_t || (tin == last_t && p <= last_p)) continue;  // visited in an earlier pass
    float t = tin, e = tref;
    int pp = p;
    list_insert(ct, ce, cp, t, e, pp);
    over_t = fminf(over_t, t);
  }
}

// LIST: the parts come from an image tile's list (tile_words, tile_count)
// unless tile_count is kTileOpen.
template <bool STATS, int BLOCK, bool GRID, bool LIST>
__device__ void trace_ray_f32(const RayW &r, bool active, uint32_t flags, int P, int NC,
                              const PartHot *__restrict__ hot, const PartAux *__restrict__ aux,
                              const Cluster *__restrict__ cl, const int32_t *__restrict__ order, const Tables *tab,
                              uint32_t stop, int top_levels, uint2 *stk, CertState &st, Contenders &con,
                              unsigned int &err,
                              Counters &cnt,
                              bool reuse, uint32_t prev_part, const uint8_t *__restrict__ dirty, bool &reused,
                              const SceneGrid *grid, uint32_t *mbox, int mwords, uint32_t tile_words,
                              uint32_t tile_count) {
  reused = false;
  st.lo1 = st.hi1 = st.te1 = st.lo2 = st.hi_min = Num<float>::inf();
  st.part1 = kMissPart;
  st.cert1 = 0;
  st.vox1 = kMissVoxel;
  con.n = 0;
  con.overflow = false;
  const bool cull = (flags & SVO_TRACE_CULL) != 0;
  const bool sort = (flags & SVO_TRACE_SORT) != 0;
  if (cull && sort) {
    // Passes are warp-uniform (every lane of the warp calls this function for
    // one ray each): a lane that needs no further pass takes part with
    // need = false, so every vote below runs with the full warp mask.
    float last_t = -Num<float>::inf();
    int last_p = -1;
    bool need = active;
    if (GRID && grid != nullptr && grid->valid != 0) {  // warp-uniform: one item per warp, one tile's list
      // a ray the walk cannot take safely goes on to the cluster level below
      const SceneGrid &g = *grid;
      const bool walked = grid_walk<STATS, BLOCK>(r, need, g, g.cell_start, g.cell_parts, hot, aux, tab, stop,
                                                  top_levels, stk, mbox, mwords, st, con, err, cnt);
      if (STATS && need && walked) ++cnt.passes;
      need = need && !walked;
    }
    while (__any_sync(0xffffffffu, need)) {
      float ct[kCap], ce[kCap];
      int cp[kCap];
#pragma unroll
      for (int i = 0; i < kCap; ++i) {
        ct[i] = Num<float>::inf();
        ce[i] = 0.f;
        cp[i] = 0x7fffffff;
      }
      float over_t = Num<float>::inf();  // smallest entry that did not fit the list
      if (STATS && need) ++cnt.passes;
      if (LIST && tile_count != kTileOpen)
        cull_listed(r, need, tile_words, tile_count, hot, last_t, last_p, ct, ce, cp, over_t);
      else
        cull_pass<STATS>(r, need, NC, hot, cl, order, last_t, last_p, ct, ce, cp, over_t, cnt);
      // hit buffer reuse (Sec. IV-C, Fig. 5).  The paper reuses a pixel whose
      // ray meets one sphere, that of its unmoved previous part.  The same
      // holds whenever every part whose sphere the ray meets is unmoved and
      // so is the previous winner (or there was none): unmoved parts keep
      // their spheres and their closest leaves along the ray, so the
      // candidates are a subset of the previous ones, and they contain the
      // previous winner, whose sphere is still met.
      if (need && reuse && last_p < 0 && ct[0] != Num<float>::inf() && over_t == Num<float>::inf() &&
          (prev_part == kMissPart || (prev_part < (uint32_t)P && dirty[prev_part] == 0))) {
        bool clean = true;
#pragma unroll
        for (int i = 0; i < kCap; ++i)
          if (ct[i] != Num<float>::inf()) clean = clean && dirty[cp[i]] == 0;
        if (clean) {
          reused = true;
          need = false;
        }
      }
      if (need) {
        // visit in order of sphere entry, stop once the best hit is nearer
        bool stopped = false;
        while (ct[0] != Num<float>::inf()) {
          const float tin = ct[0], eta = ce[0];
          const int p = cp[0];
#pragma unroll
          for (int i = 0; i < kCap - 1; ++i) {
            ct[i] = ct[i + 1];
            ce[i] = ce[i + 1];
            cp[i] = cp[i + 1];
          }
          ct[kCap - 1] = Num<float>::inf();
          if (tin > prune_bound(st, r.tmax)) {
            stopped = true;
            break;
          }
          trace_part_f32<STATS, BLOCK>(r, hot[p], aux[p], eta, (uint32_t)p, tab, stop, top_levels, stk,
                                                  st, con, err, cnt);
          last_t = tin;
          last_p = p;
        }
        // another pass only if some candidate did not fit the list and may still matter
        need = !stopped && over_t < Num<float>::inf() && over_t <= prune_bound(st, r.tmax);
      }
    }
  } else {
    for (int p = 0; p < P; ++p) {
      float tin, tref = r.tmin;
      if (!active) continue;
      if (STATS) ++cnt.parts_tested;
      const bool h = part_cull(r, hot[p], tin, tref);
      if (cull && !h) continue;
      // the plain trace descends every part, even one whose sphere is missed
      trace_part_f32<STATS, BLOCK>(r, hot[p], aux[p], tref, (uint32_t)p, tab, stop, top_levels, stk, st,
                                              con, err, cnt);
    }
  }
}

template <int NI>
__device__ __forceinline__ int find_item(const TraceLaunchT<NI> &L, unsigned long long tile) {
  int lo = 0, hi = L.n_items - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (L.items[mid].tile_begin <= tile)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ void flush_stats(svo_trace_stats *st, const Counters &c, uint32_t rays, uint32_t flagged) {
  unsigned long long v[11] = {rays, flagged, c.parts_tested, c.parts_entered, c.nodes, c.leaves, c.passes,
                              c.f_winner, c.f_overlap, c.f_width, c.reused};
#pragma unroll
  for (int i = 0; i < 11; ++i) {
    unsigned long long x = v[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    v[i] = x;
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&st->rays, v[0]);
    atomicAdd(&st->flagged, v[1]);
    atomicAdd(&st->parts_tested, v[2]);
    atomicAdd(&st->parts_entered, v[3]);
    atomicAdd(&st->nodes_visited, v[4]);
    atomicAdd(&st->leaves_tested, v[5]);
    atomicAdd(&st->passes, v[6]);
    atomicAdd(&st->flag_winner, v[7]);
    atomicAdd(&st->flag_overlap, v[8]);
    atomicAdd(&st->flag_width, v[9]);
    atomicAdd(&st->reused, v[10]);
  }
}

// The ray of `lane` in pass j of warp tile `tile` of item I: its index in the
// item's ray buffer (through the item's visiting order, if any); in_range is
// false past the item's end.  The tile of an image item is a block of
// 8 x 4*rays_per_lane pixels, claimed in the item's tile order (row by row
// without one).
template <int NI>
__device__ __forceinline__ unsigned long long tile_ray(const TraceLaunchT<NI> &L, const TraceItem &I,
                                                       unsigned long long tile, int j, int lane, bool &in_range) {
  const int rpl = L.rays_per_lane;
  const unsigned long long base = (tile - I.tile_begin) * (unsigned long long)(32 * rpl);
  unsigned long long slot_i = base + (unsigned long long)(j * 32 + lane);
  in_range = slot_i < I.n;
  if (I.tiles_x) {
    const uint32_t T = (uint32_t)(tile - I.tile_begin);
    uint32_t ty, tx;
    if (I.tile_order) {
      const uint32_t v = __ldg(&I.tile_order[T]);
      tx = v & 0xFFFFu;
      ty = v >> 16;
    } else {
      ty = T / I.tiles_x;
      tx = T - ty * I.tiles_x;
    }
    const uint32_t k = (uint32_t)(j * 32 + lane);
    const uint32_t x = tx * 8u + (k & 7u);
    const unsigned long long y = (unsigned long long)ty * (unsigned long long)(4 * rpl) + (k >> 3);
    slot_i = y * I.width + x;
    in_range = x < I.width && slot_i < I.n;
  }
  return (in_range && I.perm) ? (unsigned long long)I.perm[slot_i] : slot_i;
}

// Ray `ray` of item I (in_range false: an empty ray).  Returns whether it
// takes part: a ray needs a direction (Eq. 1) -- its largest component
// magnitude must lie in [2^-60, 2^60], so that |d|^2 is a normal FP32 number
// -- and origin, direction and bounds must be numbers, with tmin <= tmax;
// anything else is a miss.  Exact comparisons: the rule does not depend on
// rounding.
__device__ __forceinline__ bool load_ray(const TraceItem &I, unsigned long long ray, bool in_range, RayW &r) {
  bool active = in_range;
  if (active) {
    const float4 o = __ldcs(&I.rays[2 * ray]);
    const float4 d = __ldcs(&I.rays[2 * ray + 1]);
    r.ox = o.x;
    r.oy = o.y;
    r.oz = o.z;
    r.tmin = o.w;
    r.dx = d.x;
    r.dy = d.y;
    r.dz = d.z;
    r.tmax = d.w;
    const float dd = d.x * d.x + d.y * d.y + d.z * d.z;
    const float dm = fmaxf(fmaxf(fabsf(d.x), fabsf(d.y)), fabsf(d.z));
    const bool finite = isfinite(o.x) && isfinite(o.y) && isfinite(o.z) && isfinite(d.x) && isfinite(d.y) &&
                        isfinite(d.z) && !isnan(o.w) && !isnan(d.w) && dm >= 0x1p-60f && dm <= 0x1p60f;
    r.inv_dd = __frcp_rn(dd);  // the correctly rounded 1 / dd
    r.inv_len = rsqrtf(dd);
    r.onorm = fmaxf(fmaxf(fabsf(o.x), fabsf(o.y)), fabsf(o.z));
    active = finite && (o.w <= d.w);
  } else {
    r.ox = r.oy = r.oz = r.dx = r.dy = r.dz = 0.f;
    r.tmin = 0.f;
    r.tmax = -1.f;
    r.inv_dd = 0.f;
    r.inv_len = 0.f;
    r.onorm = 0.f;
  }
  return active;
}

// The result of one ray, called by every lane of the warp (in_range false: a
// lane without a ray): the hit and its flags, and -- with FP64_FIX -- the
// ray's entry in the FP64 pass's list with the leaves that pass needs.
// LANE: a lane alone (its warp's other lanes are elsewhere in their work):
// its list slot and pool entries come from atomics of its own instead of
// one atomic per warp.
template <int NI, bool STATS, bool LANE = false>
__device__ __forceinline__ void finish_ray(const TraceLaunchT<NI> &L, const TraceItem &I, int it,
                                           unsigned long long ray, bool in_range, bool reused, const RayW &r,
                                           const PartAux *__restrict__ aux, const CertState &st,
                                           const Contenders &con, int lane, unsigned int &err, Counters &cnt,
                                           uint32_t &n_flag) {
  bool flagged = false, ids_ok = true;
  uint32_t tbound = 0;  // T_REFINED: the certified error exponent, biased (flag bits 8-15)
  if (in_range && reused) {
    if (I.ray_flags) I.ray_flags[ray] = SVO_RAY_REUSED;
    if (STATS) ++cnt.reused;
  } else if (in_range) {
    float t = Num<float>::inf();
    uint32_t part = kMissPart;
    unsigned long long vox = kMissVoxel;
    if (st.part1 != kMissPart) {
      // the reported t lies in [lo1, hi1]; its error is at most half the width
      const float scale = fmaxf(st.lo1, aux[st.part1].hdiag * r.inv_len);
      const bool w_ok = st.cert1 != 0u;
      const bool o_ok = st.lo2 > st.hi1;
      const bool t_ok = 0.5f * (st.hi1 - st.lo1) <= kTau * scale;
      ids_ok = w_ok && o_ok;
      flagged = !(ids_ok && t_ok);
      if (ids_ok && !t_ok && I.ray_flags) {
        // the written t and the exact one both lie in [lo1, hi1]: their
        // distance is at most 2^e scale with e = ceil(log2((hi1 - lo1) /
        // scale)), both operations rounded up
        const uint32_t bits = __float_as_uint(__fdiv_ru(__fsub_ru(st.hi1, st.lo1), scale));
        const int e = (int)(bits >> 23) - 127 + ((bits & 0x7FFFFFu) != 0u ? 1 : 0);
        tbound = (uint32_t)min(max(e + 128, 1), 255);
      }
      if (STATS) {
        cnt.f_winner += w_ok ? 0u : 1u;
        cnt.f_overlap += (w_ok && !o_ok) ? 1u : 0u;
        cnt.f_width += (ids_ok && !t_ok) ? 1u : 0u;
      }
      t = fminf(fmaxf(st.te1, st.lo1), st.hi1);
      if (!st.cert1) t = st.te1;
      part = st.part1;
      vox = st.vox1;
    }
    uint4 hv;
    hv.x = __float_as_uint(t);
    hv.y = part;
    hv.z = (uint32_t)(vox & 0xFFFFFFFFull);
    hv.w = (uint32_t)(vox >> 32);
    __stcs(&I.hits[ray], hv);
    if (I.ray_flags)
      I.ray_flags[ray] = !ids_ok ? SVO_RAY_UNCERTAIN : (flagged ? (SVO_RAY_T_REFINED | (tbound << 8)) : 0u);
    if (STATS && !ids_ok) ++n_flag;
  }
  // compact flagged rays for the FP64 pass: one list slot each and, from
  // a pool, exactly the leaves the pass needs (one atomic per warp for
  // each): the winner alone when only t needs FP64, the contenders still
  // in play (lo <= hi_min) otherwise, or -- when the contender list
  // overflowed -- one entry carrying hi_min, where the full re-trace may
  // stop.  A ray the pool cannot hold is re-traced without that bound.
  if (L.flags & SVO_TRACE_FP64_FIX) {
    const unsigned int m = LANE ? (flagged ? 1u : 0u) : __ballot_sync(0xffffffffu, flagged);
    if (m) {
      unsigned int ncon = 0;  // contenders in play
      if (flagged && !ids_ok && !con.overflow)
        for (int q = 0; q < con.n; ++q) ncon += (con.lo[q] <= st.hi_min) ? 1u : 0u;
      const unsigned int need = !flagged ? 0u : (ids_ok || con.overflow || ncon == 0u) ? 1u : ncon;
      unsigned long long slot = 0, off = 0;
      if (LANE) {
        slot = atomicAdd(L.fix_count, 1u);
        off = atomicAdd(L.cand_count, need);
      } else {
        const int leader = __ffs(m) - 1;
        unsigned int incl = need;  // inclusive scan of the lanes' pool entries
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned int v = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += v;
        }
        const unsigned int total = __shfl_sync(0xffffffffu, incl, 31);
        unsigned int basei = 0, basep = 0;
        if (lane == leader) {
          basei = atomicAdd(L.fix_count, (unsigned int)__popc(m));
          basep = atomicAdd(L.cand_count, total);
        }
        basei = __shfl_sync(0xffffffffu, basei, leader);
        basep = __shfl_sync(0xffffffffu, basep, leader);
        slot = basei + __popc(m & ((1u << lane) - 1u));
        off = (unsigned long long)basep + (incl - need);
      }
      if (flagged) {
        if (slot < L.fix_capacity) {
          const bool stored = off + need <= L.cand_capacity;
          unsigned long long nc = 0;  // leaves listed; 0 = full FP64 re-trace
          if (stored) {
            if (ids_ok) {
              // ids certified, only t needs FP64: the winner alone
              L.fix_cand[off] = make_uint4(st.part1, (uint32_t)(st.vox1 & 0xFFFFFFFFull),
                                           (uint32_t)(st.vox1 >> 32), __float_as_uint(st.lo1));
              nc = 1;
            } else if (!con.overflow && ncon > 0u) {
              for (int q = 0; q < con.n; ++q) {
                if (!(con.lo[q] <= st.hi_min)) continue;
                L.fix_cand[off + nc] = make_uint4(con.part[q], (uint32_t)(con.vox[q] & 0xFFFFFFFFull),
                                                  (uint32_t)(con.vox[q] >> 32), __float_as_uint(con.lo[q]));
                ++nc;
              }
            } else {
              // the re-trace may stop at hi_min, an upper bound (rounded up) of the winner's t
              L.fix_cand[off] = make_uint4(0u, 0u, 0u, __float_as_uint(st.hi_min));
            }
          }
          L.fix_off[slot] = stored ? (uint32_t)off : kNoCand;
          const unsigned long long t_only = ids_ok ? 1ull : 0ull;  // ids certain, t needs FP64
          L.fix_list[slot] = (nc << 48) | (t_only << 47) | ((unsigned long long)it << kRayBits) | ray;
        } else {
          err |= kErrFixOverflow;
        }
      }
    }
  }

}

// REUSE: hit buffer reuse compiled in (a separate instantiation, so that the
// common kernel carries none of its registers or tests).
// GRID: the scene-level grid walk compiled in (likewise).
// TOP: the top levels of every part staged in shared memory (a separate
// instantiation: the staged-node base is one more live register, which the
// common kernel does not carry).
// LIST: only the image tiles k_tile_cull queued, each with its parts; with GRID
// the tiles without a list walk the grid.
// IMAGE: every item's rays are image tiles (the same code at more registers).
template <int NI, bool STATS, int BLOCK, bool REUSE, bool GRID, bool TOP = false, bool LIST = false, bool IMAGE = false>
__global__ void __launch_bounds__(BLOCK, (STATS || REUSE || GRID ? 512 : LIST ? kListThreadsPerSM : IMAGE ? kImageThreadsPerSM : kTraceThreadsPerSM) / BLOCK) k_trace(const __grid_constant__ TraceLaunchT<NI> L) {
  extern __shared__ __align__(16) unsigned char smem[];
  // [tables | traversal stacks, level-major | staged part tables]
  Tables *tab = reinterpret_cast<Tables *>(smem);
  uint2 *sStack = reinterpret_cast<uint2 *>(smem + kTablesBytes) + threadIdx.x;
  const int sp = L.one_scene ? L.items[0].n_parts : 0;
  const int sc = L.one_scene ? L.items[0].n_clusters : 0;
  PartHot *sHot = reinterpret_cast<PartHot *>(smem + kTablesBytes + (size_t)L.stack_levels * BLOCK * sizeof(uint2));
  PartAux *sAux = reinterpret_cast<PartAux *>(sHot + sp);
  Cluster *sCl = reinterpret_cast<Cluster *>(sAux + sp);
  int32_t *sOrd = reinterpret_cast<int32_t *>(sCl + sc);
  uint2 *sTop = reinterpret_cast<uint2 *>(sOrd + sp + (sp & 1));  // 8-byte aligned: sOrd starts so
  const int ntop_all = (TOP && L.one_scene) ? L.top_nodes : 0;
  uint32_t *sMbox = reinterpret_cast<uint32_t *>(sTop + ntop_all) + threadIdx.x;  // word-major, stride BLOCK
  const uint32_t sTopAddr = (uint32_t)__cvta_generic_to_shared(sTop);
  load_tables(tab);
  wait_for_previous();
  if (L.gate && *L.gate_count < L.gate) return;  // the wavefront shape's launches have the rays
  if (L.one_scene) {
    const TraceItem &I0 = L.items[0];
    for (int i = threadIdx.x; i < I0.n_parts; i += BLOCK) {
      sHot[i] = I0.hot[i];
      PartAux a = I0.aux[i];
      if (ntop_all > 0) {
        const int2 t = L.top[i];
        a.spare0 = __uint_as_float((uint32_t)t.x);
        a.spare1 = __uint_as_float((uint32_t)t.y);  // count (the kernel needs only the first)
      }
      sAux[i] = a;
      sOrd[i] = I0.order[i];
    }
    for (int i = threadIdx.x; i < I0.n_clusters; i += BLOCK) sCl[i] = I0.clusters[i];
    // every part's top levels: breadth first, they are the first nodes of its array
    for (int p = 0; p < I0.n_parts && ntop_all > 0; ++p) {
      const int2 t = L.top[p];
      const uint2 *src = I0.aux[p].nodes;
      for (int k = threadIdx.x; k < t.y; k += BLOCK) sTop[t.x + k] = __ldg(&src[k]);
    }
  }
  __syncthreads();  // the only block barrier: warps then take tiles independently
  unsigned int err = 0;
  Counters cnt = {0, 0, 0, 0, 0, 0, 0, 0};
  uint32_t n_rays = 0, n_flag = 0;
  const int lane = threadIdx.x & 31;
  const unsigned long long n_tiles = LIST ? min((unsigned long long)*L.tile_count, L.n_tiles) : L.n_tiles;
  const SceneGrid *ready = nullptr;  // the grid this warp last found ready
  for (;;) {
    unsigned long long tile = 0;
    if (lane == 0) tile = atomicAdd(L.tile_counter, 1ull);
    tile = __shfl_sync(0xffffffffu, tile, 0);
    if (tile >= n_tiles) break;
    uint32_t words = 0, count = kTileOpen;
    if (LIST) {  // the queued tile and its parts: lane i holds word i & 15 of the entry
      words = reinterpret_cast<const uint32_t *>(L.tiles + tile)[lane & 15];
      tile = __shfl_sync(0xffffffffu, words, 0);
      count = __shfl_sync(0xffffffffu, words, 1);
    }
    const int it = find_item(L, tile);
    const TraceItem &I = L.items[it];
    const int P = I.n_parts, NC = I.n_clusters;
    const bool staged = L.one_scene != 0;
    const PartHot *hot = staged ? sHot : I.hot;
    const PartAux *aux = staged ? sAux : I.aux;
    const Cluster *cls = staged ? sCl : I.clusters;
    const int32_t *ord = staged ? sOrd : I.order;
    const SceneGrid *grid = nullptr;  // warp-uniform
    if (GRID && I.grid != nullptr && (!LIST || count == kTileOpen)) {
      if (ready != I.grid && __all_sync(0xffffffffu, grid_ready(I.grid))) ready = I.grid;
      if (ready == I.grid) grid = ready;
    }
    const int rpl = L.rays_per_lane;
#pragma unroll 1
    for (int j = 0; j < rpl; ++j) {
      bool in_range = false;
      const unsigned long long ray = tile_ray(L, I, tile, j, lane, in_range);
      RayW r;
      const bool active = load_ray(I, ray, in_range, r);
      if (STATS && in_range) ++n_rays;
      CertState st;
      Contenders con;
      const bool reuse = REUSE && active;
      const uint32_t prev_part = reuse ? reinterpret_cast<const uint32_t *>(&I.hits[ray])[1] : kMissPart;
      bool reused;
      trace_ray_f32<STATS, BLOCK, GRID, LIST>(r, active, L.flags, P, NC, hot, aux, cls, ord, tab, sTopAddr,
                                              (TOP && ntop_all > 0) ? L.top_levels : 0, sStack, st, con,
                                              err, cnt, reuse, prev_part, I.dirty, reused, grid,
                                              sMbox, L.mbox_words, words, count);
      finish_ray<NI, STATS>(L, I, it, ray, in_range, reused, r, aux, st, con, lane, err, cnt, n_flag);
    }
  }
  if (STATS) flush_stats(L.stats, cnt, n_rays, n_flag);
  if (err) atomicOr(L.err, err);
}

// The culling launch of SVO_TRACE_WAVEFRONT: each ray's first culling pass
// (Sec. IV-A/B), after which the ray's miss is written -- no part sphere met:
// the result the trace would write -- or the ray is queued with its
// candidates in its item's region of the queue (one atomic per warp).  The
// descent launch traces the queued rays from there.
//
// The pass goes through the scene grid where the scene has one that lists few
// parts a cell, else through the clusters.  The tables it reads (part
// spheres, and the grid's cells or the clusters' order) are staged in shared
// memory: once where the launch has one item, whose tiles the warps then
// claim; else per run of cull_chunk tiles that a block claims, whose warps
// take them from a counter in shared memory.
//
// Bound by instruction issue, with walks of different lengths (7 of 32 lanes
// at work in an instruction).  Measured against the cluster level: 1 M rays
// inside 1024 parts 0.661 -> 0.219 ms and 0.028 to build the grid (0.262 with
// the grid read through L1), 64 scenes of 4 to 256 parts, 10.9 M rays
// 1.154 -> 1.017 and 0.014.
constexpr int kCullThreads = 256;
constexpr int kCullThreadsPerSM = 768;  // 80 registers: few spills
constexpr int kCullWarps = kCullThreads / 32;

struct CullTables {
  const float4 *sphere;    // grid: by part; clusters: in the clusters' order
  const uint16_t *cstart, *cparts;
  const SceneGrid *grid;   // nullptr: by the clusters
  const GridDims *dims;
};

// Dynamic shared memory: spheres, then the grid's cell starts and part lists.
__host__ __device__ inline size_t cull_smem_bytes(int max_parts, int max_cells) {
  return (size_t)kCullWarps * kPackRing * sizeof(int2) + (size_t)max_parts * sizeof(float4) +
         (size_t)(max_cells + 1 + (max_cells & 1 ? 0 : 1) + kGridSparse * max_cells) * sizeof(uint16_t);
}

// Called by the whole block; usable: the block's shared word for its verdict
// on the grid, which other streams' builds may be about to change.
template <int NI, bool STATS>
__device__ __forceinline__ CullTables cull_stage(const TraceItem &I, unsigned char *smem, GridDims *dims, int *usable) {
  float4 *sphere = reinterpret_cast<float4 *>(smem);
  CullTables t;
  const SceneGrid *g = STATS ? nullptr : I.grid;
  if (g != nullptr) {
    if (threadIdx.x == 0) *usable = grid_ready(g) && g->valid != 0 && g->sparse != 0;
    __syncthreads();
    if (!*usable) g = nullptr;
  }
  t.grid = g;
  const float4 *src = t.grid ? I.sphere : I.sph;
  for (int i = threadIdx.x; i < I.n_parts; i += kCullThreads) sphere[i] = src[i];
  uint16_t *cstart = reinterpret_cast<uint16_t *>(sphere + I.n_parts), *cparts = cstart;
  if (t.grid) {
    const int cells = g->G * g->G * g->G, total = g->cell_start[cells];
    cparts = cstart + cells + 1;
    for (int i = threadIdx.x; i <= cells; i += kCullThreads) cstart[i] = (uint16_t)g->cell_start[i];
    for (int i = threadIdx.x; i < total; i += kCullThreads) cparts[i] = (uint16_t)g->cell_parts[i];
  }
  if (t.grid && threadIdx.x == 0) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      dims->lo[a] = g->lo[a];
      dims->cs[a] = g->cs[a];
    }
    dims->stride[0] = 1;
    dims->stride[1] = g->G;
    dims->stride[2] = g->G * g->G;
  }
  t.sphere = sphere;
  t.cstart = cstart;
  t.cparts = cparts;
  t.dims = dims;
  return t;
}

__device__ __forceinline__ void clear_list(float (&ct)[kCap], float (&ce)[kCap], int (&cp)[kCap]) {
#pragma unroll
  for (int i = 0; i < kCap; ++i) {
    ct[i] = Num<float>::inf();
    ce[i] = 0.f;
    cp[i] = 0x7fffffff;
  }
}

// The result of the lanes' first passes (done: this lane has one, active: its
// ray is one): the miss of a ray without candidates -- over_t is set only by
// a full list, so an empty list means none at all -- or its queue entry.
// Called by the whole warp.
template <int NI>
__device__ __forceinline__ void cull_finish(const TraceLaunchT<NI> &L, const TraceItem &I, int it, bool done,
                                            bool active, unsigned long long ray, const float (&ct)[kCap],
                                            const float (&ce)[kCap], const int (&cp)[kCap], float over_t) {
  const int lane = threadIdx.x & 31;
  const bool queued = done && active && ct[0] != Num<float>::inf();
  if (done && !queued) {
    __stcs(&I.hits[ray], make_uint4(0x7f800000u, kMissPart, 0xFFFFFFFFu, 0xFFFFFFFFu));
    if (I.ray_flags) I.ray_flags[ray] = 0u;
  }
  const unsigned int m = __ballot_sync(0xffffffffu, queued);
  if (m) {
    const int leader = __ffs(m) - 1;
    unsigned int base = 0;
    if (lane == leader) base = atomicAdd(&L.queue_count[it], (unsigned int)__popc(m));
    base = __shfl_sync(0xffffffffu, base, leader);
    const unsigned long long at = base + (unsigned long long)__popc(m & ((1u << lane) - 1u));
    if (queued && at >= I.n) atomicOr(L.err, kErrShared);  // another launch counted here as well
    if (queued && at < I.n) {
      QueueEntry *q = L.queue + I.qbase + at;
      q->id = make_uint4((uint32_t)ray, (uint32_t)(ray >> 32), __float_as_uint(over_t), 0u);
      q->ct = make_float4(ct[0], ct[1], ct[2], ct[3]);
      q->ce = make_float4(ce[0], ce[1], ce[2], ce[3]);
      q->cp = make_int4(cp[0], cp[1], cp[2], cp[3]);
    }
  }
}

// The tiles [tile, end) by the clusters, 32 rays at a time.
template <int NI, bool STATS>
__device__ __forceinline__ void cull_by_clusters(const TraceLaunchT<NI> &L, const TraceItem &I, int it,
                                                 unsigned long long tile, unsigned long long end,
                                                 const float4 *sph, int2 *ring, Counters &cnt, uint32_t &n_rays) {
  const int lane = threadIdx.x & 31;
  for (; tile < end; ++tile) {
#pragma unroll 1
    for (int j = 0; j < L.rays_per_lane; ++j) {
      bool in_range;
      const unsigned long long ray = tile_ray(L, I, tile, j, lane, in_range);
      RayW r;
      const bool active = load_ray(I, ray, in_range, r);
      if (STATS && in_range) ++n_rays;
      float ct[kCap], ce[kCap];
      int cp[kCap];
      clear_list(ct, ce, cp);
      float over_t = Num<float>::inf();
      if (STATS && active) ++cnt.passes;
      cull_first_packed<STATS>(r, active, I.n_clusters, sph, I.clusters, I.order, ring, ct, ce, cp, over_t, cnt);
      cull_finish(L, I, it, in_range, active, ray, ct, ce, cp, over_t);
    }
  }
}

// The tiles [tile, end) by the grid, 32 rays at a time.  (Lanes that took the
// next ray as their walk ended, twelve or more at a time, were slower: entering
// the grid costs as much as several cells, and was then run for few lanes.)
template <int NI>
__device__ __forceinline__ void cull_by_grid(const TraceLaunchT<NI> &L, const TraceItem &I, int it,
                                             unsigned long long tile, unsigned long long end, const CullTables &t,
                                             int2 *ring, Counters &cnt) {
  const int lane = threadIdx.x & 31;
  for (; tile < end; ++tile) {
#pragma unroll 1
    for (int j = 0; j < L.rays_per_lane; ++j) {
      bool in_range, ok = true;
      const unsigned long long ray = tile_ray(L, I, tile, j, lane, in_range);
      RayW r;
      const bool active = load_ray(I, ray, in_range, r);
      float ct[kCap], ce[kCap], over_t = Num<float>::inf();
      int cp[kCap];
      clear_list(ct, ce, cp);
      GridCull w;
      bool walking = active && grid_cull_start(r, *t.grid, t.cstart, w, ok);
      while (walking) walking = grid_cull_step(r, *t.dims, t.cstart, t.cparts, t.sphere, w, ct, ce, cp, over_t);
      if (__any_sync(0xffffffffu, active && !ok))  // rays the walk cannot take: the clusters
        cull_first_packed<false>(r, active && !ok, I.n_clusters, I.sph, I.clusters, I.order, ring, ct, ce, cp, over_t,
                                 cnt);
      cull_finish(L, I, it, in_range, active, ray, ct, ce, cp, over_t);
    }
  }
}

template <int NI, bool STATS>
__global__ void __launch_bounds__(kCullThreads, kCullThreadsPerSM / kCullThreads) k_cull(const __grid_constant__ TraceLaunchT<NI> L) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long sChunk;
  __shared__ unsigned int sNext;
  __shared__ int sUsable;
  __shared__ GridDims sDims;
  // [per-warp rings of member-test pairs | tables]
  int2 *ring = reinterpret_cast<int2 *>(smem) + (threadIdx.x >> 5) * kPackRing;
  unsigned char *tables = smem + kCullWarps * kPackRing * sizeof(int2);
  Counters cnt = {0, 0, 0, 0, 0, 0, 0, 0};
  uint32_t n_rays = 0;
  const int lane = threadIdx.x & 31;
  wait_for_previous();
  if (L.gate && *L.gate_count >= L.gate) return;  // the single launch traces every ray
  int staged = -1;
  CullTables t = {nullptr, nullptr, nullptr, nullptr, nullptr};
  if (L.same_scene && L.n_items == 1) {
    t = cull_stage<NI, STATS>(L.items[0], tables, &sDims, &sUsable);
    __syncthreads();
    // every warp claims its tiles for itself, one at a time while the counter keeps up (one claim a ns)
    const unsigned long long run = L.n_tiles <= 65536ull ? 1ull : 4ull;
    const auto claim = [&](unsigned long long &tile, unsigned long long &end) {
      unsigned long long k = 0;
      if (lane == 0) k = atomicAdd(L.tile_counter, run);
      tile = min(__shfl_sync(0xffffffffu, k, 0), L.n_tiles);
      end = min(tile + run, L.n_tiles);
    };
    unsigned long long tile, end;
    for (claim(tile, end); tile < end; claim(tile, end)) {
      if (!STATS && t.grid)
        cull_by_grid(L, L.items[0], 0, tile, end, t, ring, cnt);
      else
        cull_by_clusters<NI, STATS>(L, L.items[0], 0, tile, end, t.sphere, ring, cnt, n_rays);
    }
  } else {
    for (;;) {
      __syncthreads();  // the last chunk's claim is read
      if (threadIdx.x == 0) sChunk = atomicAdd(L.tile_counter, (unsigned long long)L.cull_chunk);
      __syncthreads();
      unsigned long long tile0 = sChunk;
      if (tile0 >= L.n_tiles) break;
      const unsigned long long last = min(tile0 + (unsigned long long)L.cull_chunk, L.n_tiles);
      while (tile0 < last) {  // the chunk's part of one item after another
        const int it = find_item(L, tile0);
        const TraceItem &I = L.items[it];
        const unsigned long long stop = min(last, it + 1 < L.n_items ? L.items[it + 1].tile_begin : L.n_tiles);
        __syncthreads();  // every warp is done with the last tables and the last counter
        if (threadIdx.x == 0) sNext = 0;
        if (it != staged) t = cull_stage<NI, STATS>(I, tables, &sDims, &sUsable);
        staged = it;
        __syncthreads();
        const auto claim = [&](unsigned long long &tile, unsigned long long &end) {
          unsigned int k = 0;
          if (lane == 0) k = atomicAdd(&sNext, 1u);
          tile = min(tile0 + __shfl_sync(0xffffffffu, k, 0), stop);
          end = min(tile + 1, stop);
        };
        unsigned long long tile, end;
        for (claim(tile, end); tile < end; claim(tile, end)) {
          if (!STATS && t.grid)
            cull_by_grid(L, I, it, tile, end, t, ring, cnt);
          else
            cull_by_clusters<NI, STATS>(L, I, it, tile, end, t.sphere, ring, cnt, n_rays);
        }
        tile0 = stop;
      }
    }
  }
  if (STATS) flush_stats(L.stats, cnt, n_rays, 0u);
}

// How many of kSampleRays rays, spread evenly over the item's, meet a part
// sphere: one warp a ray, its lanes over the parts.  A few us for fewer than
// 128 parts, against the culling launch's 60 to 120 on a million rays, which
// told the same but was thrown away where most rays meet a part.
__global__ void __launch_bounds__(256) k_sample(const __grid_constant__ TraceLaunchT<1> L) {
  const TraceItem &I = L.items[0];
  const int lane = threadIdx.x & 31;
  const unsigned int warp = blockIdx.x * 8u + (threadIdx.x >> 5);
  wait_for_previous();
  RayW r;
  const bool active = load_ray(I, I.n * warp / kSampleRays, true, r);
  bool met = false;
  for (int p = lane; p < I.n_parts && active; p += 32) {
    float tin, tref;
    met = met || sphere_cull(r, I.sph[p], tin, tref);
  }
  met = __any_sync(0xffffffffu, met);
  const int n = __syncthreads_count(lane == 0 && met);
  if (threadIdx.x == 0) atomicAdd(L.gate_count, (unsigned int)n);
}

// The tile-culling launch of an image trace.  One warp takes one 8x4-pixel
// tile after another (statically strided) and bounds its rays by a cone: apex at
// one ray's origin o0, axis a along that ray, half angle theta with
// 2 sin(theta/2) <= chord, the largest distance of the unit directions from
// a, and ro, the largest distance of the origins from o0.  Then its lanes test
// 32 part spheres at a time (above kTileDirect parts: the clusters first, and
// the members of those met, four clusters to a round).  A tile no sphere
// reaches gets its misses written here; any other tile is queued with its
// parts for the trace launch, which tests only those.
//
// A sphere (c, R) is left out when its centre, v = c - o0 with x = v.a and y
// its distance from the axis, satisfies y cos(theta) - x+ sin(theta) > R' or
// -x > R' (the cone lies in both half spaces, so this is a lower bound of the
// distance), with R' = R + ro + 96 u (|v|_1 + R + ro): part_cull passes a
// sphere only when the exact line comes within R + 32 u R + 22 u |l|_1 of its
// centre, and the rest covers this test's own rounding.  So every part that
// passes part_cull for a ray of the tile is listed, and the trace launch
// finds the candidates it would find from the clusters.
//
// Why: most tiles meet few parts or none, yet every ray tested every cluster
// and the members of those it met, in a kernel held to 24 warps per SM by the
// descent's registers.  Here a tile costs two tests a lane for 64 parts, at
// 32 registers.  2.07 M rays against 1024 parts: 49 us (100 MB at 2 TB/s), and
// the trace with its tiles' lists 290 us, against 511 us through the scene
// grid and 27 us to build it; 6.7 M rays of nine requests: 92 + 790 us against
// 1165.
constexpr int kTileThreads = 256;
constexpr int kTileDirect = 64;  // parts up to which the part spheres are tested without the clusters

struct TileCone {
  float ox, oy, oz, ax, ay, az, ch, cl, ro;
};

__device__ __forceinline__ bool cone_meets(const TileCone &k, float4 s) {
  const float vx = s.x - k.ox, vy = s.y - k.oy, vz = s.z - k.oz;
  const float vn = fabsf(vx) + fabsf(vy) + fabsf(vz);
  const float x = vx * k.ax + vy * k.ay + vz * k.az;
  const float wx = fmaf(-x, k.ax, vx), wy = fmaf(-x, k.ay, vy), wz = fmaf(-x, k.az, vz);
  float y;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(wx * wx + wy * wy + wz * wz));
  const float R0 = s.w + k.ro;
  const float R = fmaf(96.0f * kU, vn + R0, R0);
  // a centre too far away for these squares, or a value that is not a number, keeps the part
  return s.w >= 0.f && (!(fmaf(y, k.cl, -fmaxf(x, 0.f) * k.ch) > R || -x > R) || vn > 1e15f);
}

template <int NI>
__global__ void __launch_bounds__(kTileThreads) k_tile_cull(const __grid_constant__ TraceLaunchT<NI> L) {
  __shared__ __align__(4) uint16_t sList[kTileThreads / 32][kTileParts];
  const int lane = threadIdx.x & 31;
  const unsigned int below = (1u << lane) - 1u;
  uint16_t *list = sList[threadIdx.x >> 5];
  wait_for_previous();
  const unsigned long long n_warps = (unsigned long long)gridDim.x * (kTileThreads / 32);
  for (unsigned long long tile = (unsigned long long)blockIdx.x * (kTileThreads / 32) + (threadIdx.x >> 5);
       tile < L.n_tiles; tile += n_warps) {
    const int it = NI > 1 ? find_item(L, tile) : 0;
    const TraceItem &I = L.items[it];
    bool in_range;
    const unsigned long long ray = tile_ray(L, I, tile, 0, lane, in_range);
    RayW r;
    const bool active = load_ray(I, ray, in_range, r);
    const unsigned int am = __ballot_sync(0xffffffffu, active);
    bool open = false;
    uint32_t cnt = 0;
    if (am) {
      TileCone k;
      const int src = ((am >> 12) & 1u) ? 12 : __ffs(am) - 1;  // lane 12: next to the tile's centre
      const float ux = r.dx * r.inv_len, uy = r.dy * r.inv_len, uz = r.dz * r.inv_len;
      k.ax = __shfl_sync(0xffffffffu, ux, src);
      k.ay = __shfl_sync(0xffffffffu, uy, src);
      k.az = __shfl_sync(0xffffffffu, uz, src);
      k.ox = __shfl_sync(0xffffffffu, r.ox, src);
      k.oy = __shfl_sync(0xffffffffu, r.oy, src);
      k.oz = __shfl_sync(0xffffffffu, r.oz, src);
      const float ex = ux - k.ax, ey = uy - k.ay, ez = uz - k.az;
      const float e2 = ex * ex + ey * ey + ez * ez;
      const float dl = fabsf(r.ox - k.ox) + fabsf(r.oy - k.oy) + fabsf(r.oz - k.oz);
      // no cone for rays that reach behind their origin or spread over more than 30 degrees
      open = __any_sync(0xffffffffu, active && (!(e2 <= 0.25f) || r.tmin < 0.f));
      // non-negative floats order as their bits do
      k.ch = sqrtf(__uint_as_float(__reduce_max_sync(0xffffffffu, active ? __float_as_uint(e2) : 0u))) * 1.0001f + 1e-6f;
      k.cl = 1.0f - 0.5f * k.ch * k.ch - 1e-6f;
      k.ro = __uint_as_float(__reduce_max_sync(0xffffffffu, active ? __float_as_uint(dl) : 0u));
      if (!open) {
        __syncwarp();  // the last tile's list is read
        if (I.n_parts <= kTileDirect) {
          for (int b = 0; b < I.n_parts; b += 32) {
            const int q = b + lane;
            const bool hit = q < I.n_parts && cone_meets(k, I.sph[q]);
            const unsigned int hm = __ballot_sync(0xffffffffu, hit);
            const uint32_t pos = cnt + __popc(hm & below);
            if (hit && pos < (uint32_t)kTileParts) list[pos] = (uint16_t)I.order[q];
            cnt += __popc(hm);
          }
        } else {
          for (int b = 0; b < I.n_clusters; b += 32) {
            const int c = b + lane;
            unsigned int cm = __ballot_sync(0xffffffffu, c < I.n_clusters && cone_meets(k, I.clusters[c].sphere));
            while (cm) {
              // lane q takes member q & 7 of the (q >> 3)-th cluster left
              int mine = -1;
#pragma unroll
              for (int g = 0; g < 4; ++g) {
                const int first = __ffs(cm) - 1;  // -1: none left
                if ((lane >> 3) == g) mine = first;
                cm &= cm - 1u;
              }
              const int q = (b + mine) * kClusterSize + (lane & 7);
              const bool hit = mine >= 0 && q < I.n_parts && cone_meets(k, I.sph[q]);
              const unsigned int hm = __ballot_sync(0xffffffffu, hit);
              const uint32_t pos = cnt + __popc(hm & below);
              if (hit && pos < (uint32_t)kTileParts) list[pos] = (uint16_t)I.order[q];
              cnt += __popc(hm);
            }
          }
        }
        __syncwarp();
      }
    }
    if (!open && cnt == 0) {
      if (in_range) {
        __stcs(&I.hits[ray], make_uint4(0x7f800000u, kMissPart, 0xFFFFFFFFu, 0xFFFFFFFFu));
        if (I.ray_flags) I.ray_flags[ray] = 0u;
      }
      continue;
    }
    const bool listed = !open && cnt <= (uint32_t)kTileParts;
    if (!listed && lane == 0 && (L.flags & SVO_TRACE_GRID) && I.grid != nullptr) *L.gate_count = 1u;
    unsigned int slot = 0;
    if (lane == 0) slot = atomicAdd(L.tile_count, 1u);
    slot = __shfl_sync(0xffffffffu, slot, 0);
    if (slot >= L.n_tiles) {  // another launch counted here as well
      if (lane == 0) atomicOr(L.err, kErrShared);
      continue;
    }
    if (lane < 16) {
      uint32_t w = (uint32_t)tile;
      if (lane == 1) w = listed ? cnt : kTileOpen;
      if (lane >= 2) w = reinterpret_cast<const uint32_t *>(list)[lane - 2];
      reinterpret_cast<uint32_t *>(L.tiles + slot)[lane] = w;
    }
  }
}

// The descent launch of SVO_TRACE_WAVEFRONT.  Every lane works through the
// queued rays on its own: when its part's descent ends it goes on to the
// ray's next candidate, a further culling pass, or the ray's result and the
// next queued ray, while the other lanes of its warp carry on with their
// own descents.  A warp thus stays full until the queue runs dry, instead
// of waiting for the longest of a tile's 32 descents (incoherent rays into
// assets of different depths descend for very different lengths).  Each
// step of the loop: lanes that need a ray take the next entries of the
// warp's claimed run (32 entries claimed with one atomic), lanes between
// parts set up their next part, and every lane in a descent takes one node.
// The arithmetic is that of the fused kernel: part_start, descent_step,
// cull_pass and finish_ray, so results are the same bit for bit.
constexpr int kRefillLanes = 16;  // lanes that wait before the warp serves them

template <int NI, bool STATS, int BLOCK>
__global__ void __launch_bounds__(BLOCK, 512 / BLOCK) k_descend(const __grid_constant__ TraceLaunchT<NI> L) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long sQE[NI + 1];  // first entry of each item in the flat order of all queued rays
  // [tables | traversal stacks, level-major | staged part tables]
  Tables *tab = reinterpret_cast<Tables *>(smem);
  uint2 *sStack = reinterpret_cast<uint2 *>(smem + kTablesBytes) + threadIdx.x;
  const int sp = L.one_scene ? L.items[0].n_parts : 0;
  const int sc = L.one_scene ? L.items[0].n_clusters : 0;
  PartHot *sHot = reinterpret_cast<PartHot *>(smem + kTablesBytes + (size_t)L.stack_levels * BLOCK * sizeof(uint2));
  PartAux *sAux = reinterpret_cast<PartAux *>(sHot + sp);
  Cluster *sCl = reinterpret_cast<Cluster *>(sAux + sp);
  int32_t *sOrd = reinterpret_cast<int32_t *>(sCl + sc);
  load_tables(tab);
  wait_for_previous();
  if (L.gate && *L.gate_count >= L.gate) return;  // the single launch traces every ray
  if (L.one_scene) {
    const TraceItem &I0 = L.items[0];
    for (int i = threadIdx.x; i < I0.n_parts; i += BLOCK) {
      sHot[i] = I0.hot[i];
      sAux[i] = I0.aux[i];
      sOrd[i] = I0.order[i];
    }
    for (int i = threadIdx.x; i < I0.n_clusters; i += BLOCK) sCl[i] = I0.clusters[i];
  }
  if (threadIdx.x == 0) {
    unsigned long long acc = 0;
    for (int i = 0; i < L.n_items; ++i) {
      sQE[i] = acc;
      acc += min((unsigned long long)L.queue_count[i], L.items[i].n);
    }
    sQE[L.n_items] = acc;
  }
  __syncthreads();  // the only block barrier
  const unsigned long long total = sQE[L.n_items];
  const bool staged = L.one_scene != 0;
  unsigned int err = 0;
  Counters cnt = {0, 0, 0, 0, 0, 0, 0, 0};
  uint32_t n_flag = 0;
  const int lane = threadIdx.x & 31;
  enum { kNeedRay = 0, kBetween = 1, kDescending = 2, kDone = 3 };
  int state = kNeedRay;
  int it = 0;
  unsigned long long ray = 0;
  RayW r;
  CertState st;
  Contenders con;
  float ct[kCap], ce[kCap];
  int cp[kCap];
  float over_t = 0.f, last_t = 0.f;
  int last_p = -1;
  bool stopped = false;
  Descent ds;
  unsigned long long wnext = 0, wend = 0;  // the warp's claimed run of entries (warp-uniform)
  for (;;) {
    // lanes waiting for work are served together, once enough of them wait
    // (or no lane is descending): the set-up of a part and the result of a
    // ray then run for many lanes at a time
    const unsigned int waiting = __ballot_sync(0xffffffffu, state == kNeedRay || state == kBetween);
    const bool serve = __popc(waiting) >= kRefillLanes || !__any_sync(0xffffffffu, state == kDescending);
    // lanes that need a ray take the next entries of the warp's run
    unsigned int want = serve ? __ballot_sync(0xffffffffu, state == kNeedRay) : 0u;
    while (want) {
      if (wnext >= wend) {
        unsigned long long b = 0;
        if (lane == 0) b = atomicAdd(L.queue_tile, 32ull);
        b = __shfl_sync(0xffffffffu, b, 0);
        wnext = b;
        wend = b + 32ull < total ? b + 32ull : total;
        if (wnext >= total) {
          if (want & (1u << lane)) state = kDone;  // the queue is empty
          break;
        }
      }
      const unsigned int take = min((unsigned int)__popc(want), (unsigned int)(wend - wnext));
      const unsigned int rank = __popc(want & ((1u << lane) - 1u));
      if ((want & (1u << lane)) && rank < take) {
        const unsigned long long g = wnext + rank;
        int lo = 0, hi = L.n_items - 1;  // the item holding flat entry g
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (sQE[mid] <= g)
            lo = mid;
          else
            hi = mid - 1;
        }
        it = lo;
        const TraceItem &I = L.items[it];
        const QueueEntry *q = L.queue + I.qbase + (g - sQE[it]);
        const uint4 id = q->id;
        ray = (unsigned long long)id.x | ((unsigned long long)id.y << 32);
        over_t = __uint_as_float(id.z);
        const float4 a = q->ct, b = q->ce;
        const int4 c = q->cp;
        static_assert(kCap == 4, "a queued ray carries four candidates");
        ct[0] = a.x, ct[1] = a.y, ct[2] = a.z, ct[3] = a.w;
        ce[0] = b.x, ce[1] = b.y, ce[2] = b.z, ce[3] = b.w;
        cp[0] = c.x, cp[1] = c.y, cp[2] = c.z, cp[3] = c.w;
        load_ray(I, ray, true, r);  // a queued ray is a ray: the culling launch checked it
        st.lo1 = st.hi1 = st.te1 = st.lo2 = st.hi_min = Num<float>::inf();
        st.part1 = kMissPart;
        st.cert1 = 0;
        st.vox1 = kMissVoxel;
        con.n = 0;
        con.overflow = false;
        last_t = -Num<float>::inf();
        last_p = -1;
        stopped = false;
        state = kBetween;
      }
      // warp-uniform bookkeeping of the run and of the lanes still waiting
      unsigned int served = 0u, w = want;
      for (unsigned int k = 0; k < take; ++k) {
        served |= w & (0u - w);  // lowest waiting lane
        w &= w - 1u;
      }
      want &= ~served;
      wnext += take;
    }
    // lanes between parts: the next candidate, a further culling pass, or the ray's result
    while (serve && state == kBetween) {
      const TraceItem &I = L.items[it];
      const PartHot *hot = staged ? sHot : I.hot;
      const PartAux *aux = staged ? sAux : I.aux;
      if (ct[0] != Num<float>::inf()) {
        const float tin = ct[0], tref = ce[0];
        const int p = cp[0];
#pragma unroll
        for (int i = 0; i < kCap - 1; ++i) {
          ct[i] = ct[i + 1];
          ce[i] = ce[i + 1];
          cp[i] = cp[i + 1];
        }
        ct[kCap - 1] = Num<float>::inf();
        if (tin > prune_bound(st, r.tmax)) {  // this and every later candidate start beyond the best hit
          stopped = true;
#pragma unroll
          for (int i = 0; i < kCap; ++i) ct[i] = Num<float>::inf();
          continue;
        }
        last_t = tin;
        last_p = p;
        if (part_start<STATS, CertState>(r, hot[p], aux[p], tref, (uint32_t)p, 0u, 0, st, ds, cnt)) state = kDescending;
        continue;
      }
      if (!stopped && over_t < Num<float>::inf() && over_t <= prune_bound(st, r.tmax)) {
        // some candidate did not fit the list and may still matter: another pass
#pragma unroll
        for (int i = 0; i < kCap; ++i) {
          ct[i] = Num<float>::inf();
          ce[i] = 0.f;
          cp[i] = 0x7fffffff;
        }
        over_t = Num<float>::inf();
        if (STATS) ++cnt.passes;
        cull_pass<STATS, false>(r, true, I.n_clusters, hot, staged ? sCl : I.clusters, staged ? sOrd : I.order,
                                       last_t, last_p, ct, ce, cp, over_t, cnt);
        continue;
      }
      finish_ray<NI, STATS, true>(L, I, it, ray, true, false, r, aux, st, con, lane, err, cnt, n_flag);
      state = kNeedRay;
    }
    if (__all_sync(0xffffffffu, state == kDone)) break;
    if (state == kDescending && !descent_step<STATS, BLOCK>(ds, sStack, tab, st, con, err, cnt))
      state = kBetween;
  }
  if (STATS) flush_stats(L.stats, cnt, 0u, n_flag);
  if (err) atomicOr(L.err, err);
}

// ------------------------------------------------- one ray by a whole warp

// The search of one ray with its node visits spread over a warp's lanes.  The
// ray's candidate parts are found 32 at a time and set up one per lane; their
// roots go onto a stack of nodes in shared memory, and every round takes up to
// 32 nodes off it, one per lane, and pushes the children the ray meets.  A
// sink takes the leaves (leaf), prunes (bound, as rel_bound) and gathers what
// the lanes found after every round (round).  A long chain of node visits --
// a grazing ray's hundreds -- takes a few dozen rounds.
//
// The stack holds kCoopStack nodes.  While it has room for what 32 nodes can
// push (at most 7 net each) a round takes 32; nearer to the end it takes
// fewer, down to one at a time, for which a depth-first search needs no more
// than 7 slots a level: the room kept back for it.
constexpr int kCoopStack = 320;
constexpr int kCoopParts = 16;  // candidate parts set up at a time
constexpr int kCoopReserve = 7 * kMaxDepth + 8;
static_assert(kCoopStack > 2 * kCoopReserve + 32, "room to work in");

struct CoopWarp {
  uint4 stack[kCoopStack];  // node | corner x, y << 16 | corner z, level << 16, part slot << 24 | entry (the part's)
  Descent part[kCoopParts];
};

// Takes the nodes off the stack (top of them, warp-uniform) until it is empty.
template <typename Sink>
__device__ __forceinline__ void coop_drain(CoopWarp &w, int top, const Tables *__restrict__ tab, Sink &sink,
                                           unsigned int &err) {
  const int lane = threadIdx.x & 31;
  while (top > 0) {
    const int n = min(top, max(1, min(32, (kCoopStack - kCoopReserve - top) / 7)));
    top -= n;
    uint4 e = make_uint4(0u, 0u, 0u, 0u);
    if (lane < n) e = w.stack[top + lane];
    __syncwarp();
    uint32_t hit = 0;  // children to push (mirrored)
    const uint32_t slot = e.z >> 24;
    Descent s = w.part[slot];
    s.X = 0x3F800000u | ((e.y & 0xFFFFu) << 7);
    s.Y = 0x3F800000u | ((e.y >> 16) << 7);
    s.Z = 0x3F800000u | ((e.z & 0xFFFFu) << 7);
    s.level = (int)((e.z >> 16) & 0xFFu);
    const NodePlanes nd(s);
    uint2 desc = make_uint2(0u, 0u);
    if (lane < n && __uint_as_float(e.w) <= sink.bound(s)) {
      desc = __ldg(&s.nodes[e.x]);
      hit = nd.hits(sink.bound(s)) & tab->mirror[s.mir][desc.y & 0xFFu];
      if (s.level == s.D - 1) {
        for (; hit != 0u; hit &= hit - 1u) {
          const uint32_t m = (uint32_t)__ffs(hit) - 1u;
          if (nd.entry(m) <= sink.bound(s)) sink.leaf(s, nd, m);
        }
      }
    }
    int at = __popc(hit);
    const int own = at;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += v;
    }
    const int total = __shfl_sync(0xffffffffu, at, 31);
    const int shift = 22 - s.level;  // the bit of a corner's float that a step down sets
    for (int pos = top + at - own; hit != 0u; ++pos) {
      const uint32_t m = 31u - (uint32_t)__clz(hit);  // the child nearest to the ray's start goes on top
      hit &= ~(1u << m);
      const uint32_t k = m ^ s.mir;
      uint32_t idx = desc.x + __popc(desc.y & ((1u << k) - 1u));
      float en = nd.entry(m);
      if (idx >= s.n_nodes) {  // not followed: no bound admits this entry
        err |= kErrNodeIndex;
        idx = 0;
        en = __int_as_float(0x7fffffff);
      }
      const uint32_t cx = ((s.X & 0x7FFFFFu) | ((m & 1u) << shift)) >> 7,
                     cy = ((s.Y & 0x7FFFFFu) | (((m >> 1) & 1u) << shift)) >> 7,
                     cz = ((s.Z & 0x7FFFFFu) | ((m >> 2) << shift)) >> 7;
      w.stack[pos] = make_uint4(idx, cx | (cy << 16), cz | ((uint32_t)(s.level + 1) << 16) | (slot << 24),
                                __float_as_uint(en));
    }
    top += total;
    __syncwarp();
    sink.round();
  }
}

// All parts of item I.  r is the same on every lane.
template <typename Sink>
__device__ __forceinline__ void coop_trace(CoopWarp &w, const TraceItem &I, const RayW &r,
                                           const Tables *__restrict__ tab, Sink &sink, unsigned int &err,
                                           Counters &cnt) {
  const int lane = threadIdx.x & 31;
  int n_cand = 0;
  for (int base = 0; base < I.n_parts; base += 32) {
    const int p = base + lane;
    Descent ds;
    float tin, tref;
    const bool in = p < I.n_parts && part_cull(r, I.hot[p], tin, tref) && !(tin > sink.best()) &&
                    part_start<false>(r, I.hot[p], I.aux[p], tref, (uint32_t)p, 0u, 0, sink, ds, cnt);
    for (unsigned int m = __ballot_sync(0xffffffffu, in); m != 0u;) {
      const int c = min(__popc(m), kCoopParts - n_cand);  // as many as there are slots left
      const int q = __popc(m & ((1u << lane) - 1u));
      if (((m >> lane) & 1u) && q < c) {
        w.part[n_cand + q] = ds;
        w.stack[n_cand + q] = make_uint4(0u, 0u, (uint32_t)(n_cand + q) << 24, __float_as_uint(ds.tmin));
      }
      n_cand += c;
      for (int k = 0; k < c; ++k) m &= m - 1u;  // the lowest c lanes are in
      __syncwarp();
      if (n_cand == kCoopParts) {
        coop_drain(w, n_cand, tab, sink, err);
        n_cand = 0;
      }
    }
  }
  coop_drain(w, n_cand, tab, sink, err);
}

// The exact search (the FP64 pass's re-trace): the FP32 search with inflated
// boxes, so no leaf the FP64 rule could hit is skipped, collects the leaves it
// reaches, and the warp decides them in FP64, 32 at a time.
constexpr int kLeafBuf = 31 + 32 * 8;  // emptied from 32 on; a round adds at most 8 a lane
struct LeafBuf {
  unsigned long long vox[kLeafBuf];
  uint32_t part[kLeafBuf];
  unsigned int n;
};

struct ExactSink {
  LeafBuf &buf;
  const TraceItem &I;
  float4 o, d;    // the ray; d.w: where the search ends
  float closest;  // upper bound of the closest hit's t so far
  ExactState ex;  // this lane's

  __device__ __forceinline__ float best() const { return closest; }
  __device__ __forceinline__ float bound(const Descent &s) const {
    return fminf(s.tmax, __fsub_ru(closest, s.tshift));
  }
  __device__ __forceinline__ void leaf(const Descent &s, const NodePlanes &, uint32_t m) {
    const unsigned int q = atomicAdd(&buf.n, 1u);
    if (q < (unsigned int)kLeafBuf) {
      buf.vox[q] = leaf_voxel(s, m);
      buf.part[q] = s.part;
    }
  }
  __device__ __forceinline__ void decide() {
    const int lane = threadIdx.x & 31, n = (int)buf.n;
    for (int k = lane; k < n; k += 32) {
      const uint32_t p = buf.part[k];
      double tq;
      if (leaf_entry64(local_ray64(I.inv64 + 12 * p, o, d), I.aux[p].depth, buf.vox[k], o.w, d.w, tq))
        offer(ex, tq, p, buf.vox[k]);
    }
    double t = ex.t;
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) t = fmin(t, __shfl_xor_sync(0xffffffffu, t, q));
    closest = __double2float_ru(t);
    __syncwarp();
    if (lane == 0) buf.n = 0;
    __syncwarp();
  }
  __device__ __forceinline__ void round() {
    if (buf.n >= 32u) decide();
    __syncwarp();  // every lane has read the count
  }
};

__device__ __forceinline__ float rel_bound(const ExactSink &s, float tmax_rel, float tshift) {
  return fminf(tmax_rel, __fsub_ru(s.closest, tshift));
}

// ------------------------------------------------------------- FP64 pass

// One warp's 32 list entries in the FP64 pass.
struct FixWarp {
  double o[3][32], inv[3][32];  // the ray in the frame of its first leaf's part
  unsigned long long key[32], vox[32];  // one round's results
  uint32_t part[32], first[32], off[32];
  float tmin[32], tmax[32];
  int depth[32], begin[32];  // begin: an entry's first place in the flat order of the other leaves
};

struct RetraceWarp {
  CoopWarp coop;
  LeafBuf buf;
};

union FixUnion {  // a warp does one or the other
  FixWarp list;
  RetraceWarp re;
};

// Lexicographic minimum of (t, part, voxel) across the warp (every lane
// returns it).
__device__ __forceinline__ void warp_min(ExactState &s) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ExactState x;
    x.t = __shfl_xor_sync(0xffffffffu, s.t, o);
    x.part = __shfl_xor_sync(0xffffffffu, s.part, o);
    x.vox = __shfl_xor_sync(0xffffffffu, s.vox, o);
    offer(s, x.t, x.part, x.vox);
  }
}

__device__ __forceinline__ void write_fixed(const TraceItem &I, unsigned long long ray, const ExactState &st,
                                            uint32_t why) {
  uint4 hv;
  hv.x = __float_as_uint((float)st.t);
  hv.y = st.part;
  hv.z = (uint32_t)(st.vox & 0xFFFFFFFFull);
  hv.w = (uint32_t)(st.vox >> 32);
  I.hits[ray] = hv;
  if (I.ray_flags) I.ray_flags[ray] = why | SVO_RAY_FIXED;
}

// Lexicographic minimum of (t, part, voxel) across each aligned group of 8
// lanes (every lane of the group returns it).
__device__ __forceinline__ void group_min8(ExactState &s) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    ExactState x;
    x.t = __shfl_xor_sync(0xffffffffu, s.t, o);
    x.part = __shfl_xor_sync(0xffffffffu, s.part, o);
    x.vox = __shfl_xor_sync(0xffffffffu, s.vox, o);
    offer(s, x.t, x.part, x.vox);
  }
}

// The FP64 pass for a flagged ray without a contender list (the list
// overflowed), called by the whole warp (i: its list index, e: its entry).
// The warp re-traces the ray together (coop_trace).  The segment ends at the
// FP32 pass's certain upper bound of the winner's t where one was stored: the
// winner (and every leaf tied with it) starts no later, so no candidate is
// lost and the leaves beyond it are never tested in FP64.  With the parts dealt
// over the lanes and each lane's leaves decided as it came to them, one such
// ray took 50 to 100 us (its node visits one after another), and the 42,600 of
// 1.05 M rays into depth-13 parts 1.73 ms.
template <int NI>
__device__ void overflow_retrace(const TraceLaunchT<NI> &L, unsigned long long i, unsigned long long e,
                                 const Tables *tab, FixUnion &u, unsigned int &err, Counters &cnt) {
  const int lane = threadIdx.x & 31;
  const uint32_t why = ((e >> 47) & 1ull) ? SVO_RAY_T_REFINED : SVO_RAY_UNCERTAIN;
  const int it = (int)((e >> kRayBits) & 0x7Fu);
  const unsigned long long ray = e & ((1ull << kRayBits) - 1ull);
  const TraceItem &I = L.items[it];
  const float4 o = I.rays[2 * ray], d = I.rays[2 * ray + 1];
  const uint32_t off = L.fix_off[i];
  const float tcap = off != kNoCand ? __uint_as_float(L.fix_cand[off].w) : Num<float>::inf();
  RayW r;
  r.ox = o.x;
  r.oy = o.y;
  r.oz = o.z;
  r.tmin = o.w;
  r.dx = d.x;
  r.dy = d.y;
  r.dz = d.z;
  r.tmax = fminf(d.w, tcap);
  r.inv_dd = 1.0f / (d.x * d.x + d.y * d.y + d.z * d.z);
  r.inv_len = 0.f;
  r.onorm = 0.f;
  ExactSink sink = {u.re.buf, I, o, make_float4(d.x, d.y, d.z, r.tmax), Num<float>::inf(),
                    {Num<double>::inf(), kMissPart, kMissVoxel}};
  __syncwarp();  // the union's other member is read
  if (lane == 0) sink.buf.n = 0;
  __syncwarp();
  coop_trace(u.re.coop, I, r, tab, sink, err, cnt);
  sink.decide();
  warp_min(sink.ex);
  if (lane == 0) write_fixed(I, ray, sink.ex, why);
}

// A candidate's t as an unsigned integer of the same order (-0 as 0), so that
// comparing candidates takes no FP64 instruction; kNoHitKey: no hit.
constexpr unsigned long long kNoHitKey = 0xFFFFFFFFFFFFFFFFull;
__device__ __forceinline__ unsigned long long order_key(double t) {
  const long long b = __double_as_longlong(t + 0.0);
  return (unsigned long long)(b ^ ((b >> 63) | (1ll << 63)));
}
__device__ __forceinline__ double key_value(unsigned long long k) {
  const long long b = (long long)k;
  return __longlong_as_double(b < 0 ? (long long)(k ^ (1ull << 63)) : ~b);
}

// Re-intersects the rays the FP32 pass flagged, in FP64 and without
// certification:
//   * with a contender list (the leaves that may still be the closest hit),
//     the contenders are intersected by the exact closed-box rule, spread
//     over lanes, and the lexicographic minimum of (t, part, voxel) kept;
//   * without one (the contender list overflowed, or the leaf pool was
//     full), the warp re-traces the ray (overflow_retrace).
// Bound by the FP64 pipes on long lists (GB300 issues FP64 at 2 lanes per
// clock and SM, whatever a warp's active lanes), by latency on short ones.
// Lists of up to two rounds of four entries per warp give each entry a group
// of eight lanes, so that they spread over the GPU; longer ones are taken 32
// entries a warp (below).  1.05 M rays into depth-13 parts (428 K t
// refinements, 289 K contender lists of 5 leaves on average, 43 K re-traces):
// 2.55 -> 1.00 ms; 116 K entries of 64 scenes 59 -> 36 us.
template <int NI>
__global__ void __launch_bounds__(kBlock) k_fix(const __grid_constant__ TraceLaunchT<NI> L) {
  __shared__ FixUnion sFix[kBlock / 32];
  // the rare re-traces read the order tables from global memory (L1/L2), so
  // blocks start without staging them
  const Tables *tab = &g_tables;
  unsigned int err = 0;
  Counters cnt = {0, 0, 0, 0, 0, 0, 0, 0};
  wait_for_previous();
  const unsigned long long n = min((unsigned long long)*L.fix_count, L.fix_capacity);
  const int lane = threadIdx.x & 31;
  const unsigned long long n_warps = (unsigned long long)gridDim.x * (blockDim.x / 32);
  const unsigned long long warp = blockIdx.x + (unsigned long long)gridDim.x * (threadIdx.x >> 5);
  // Four list entries per warp, one group of 8 lanes each (at most 16
  // contenders per entry, two per lane): FP64 issues at a few lanes per clock
  // and a warp instruction holds the pipe whatever its active lanes, so
  // packing entries cuts the pipe time per entry.  Entries without contenders
  // are re-traced afterwards by the whole warp, one at a time.
  static_assert(kContenders <= 16, "8-lane groups, two contenders per lane at most");
  const int sub = lane >> 3, sl = lane & 7;
  if (n > 8ull * n_warps) {
    // A long list (more than two rounds of four entries per warp): runs of 32
    // entries per warp, one a lane for its first leaf (every t refinement has
    // no other).  The other contenders of the 32 entries are dealt over the
    // lanes in one flat order, so that an FP64 instruction serves 32 of them
    // however they are distributed; those in the part of the entry's first leaf
    // (nearly all) reuse its local ray from shared memory.  Each entry's lane
    // then takes the minimum of its own.
    FixWarp &w = sFix[threadIdx.x >> 5].list;
    for (unsigned long long i0 = 32 * warp; i0 < n; i0 += 32 * n_warps) {
      const unsigned long long i = i0 + (unsigned long long)lane;
      const bool have = i < n;
      const unsigned long long e = have ? L.fix_list[i] : 0ull;
      const int nc = (int)(e >> 48);
      const int it = (int)((e >> kRayBits) & 0x7Fu);
      const unsigned long long ray = e & ((1ull << kRayBits) - 1ull);
      unsigned long long best = kNoHitKey, vox = kMissVoxel;
      uint32_t part = kMissPart;
      if (nc >= 1) {
        const TraceItem &I = L.items[it];
        const float4 o = I.rays[2 * ray], d = I.rays[2 * ray + 1];
        const uint32_t off = L.fix_off[i];
        const uint4 cv = L.fix_cand[off];
        const unsigned long long v = (unsigned long long)cv.y | ((unsigned long long)cv.z << 32);
        const int depth = I.aux[cv.x].depth;
        const LocalRay64 l = local_ray64(I.inv64 + 12 * cv.x, o, d);
        double tq;
        if (leaf_entry64(l, depth, v, o.w, d.w, tq)) {
          best = order_key(tq);
          part = cv.x;
          vox = v;
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          w.o[k][lane] = l.o[k];
          w.inv[k][lane] = l.inv[k];
        }
        w.tmin[lane] = o.w;
        w.tmax[lane] = d.w;
        w.first[lane] = cv.x;
        w.depth[lane] = depth;
        w.off[lane] = off;
      }
      const int more = nc >= 2 ? nc - 1 : 0;
      int begin = more;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, begin, o);
        if (lane >= o) begin += v;
      }
      const int total = __shfl_sync(0xffffffffu, begin, 31);
      begin -= more;
      w.begin[lane] = begin;
      __syncwarp();
      for (int base = 0; base < total; base += 32) {
        const int f = base + lane;
        int own = 0;  // the last entry that begins at or before f
#pragma unroll
        for (int k = 16; k > 0; k >>= 1)
          if (w.begin[own + k] <= f) own += k;
        const unsigned long long eo = __shfl_sync(0xffffffffu, e, own);
        unsigned long long key = kNoHitKey, v = kMissVoxel;
        uint32_t p = kMissPart;
        if (f < total) {
          const uint4 cv = L.fix_cand[w.off[own] + 1 + (f - w.begin[own])];
          p = cv.x;
          v = (unsigned long long)cv.y | ((unsigned long long)cv.z << 32);
          int depth = w.depth[own];
          LocalRay64 l;
          if (p == w.first[own]) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              l.o[k] = w.o[k][own];
              l.inv[k] = w.inv[k][own];
            }
          } else {
            const TraceItem &I = L.items[(int)((eo >> kRayBits) & 0x7Fu)];
            const unsigned long long ry = eo & ((1ull << kRayBits) - 1ull);
            l = local_ray64(I.inv64 + 12 * p, I.rays[2 * ry], I.rays[2 * ry + 1]);
            depth = I.aux[p].depth;
          }
          double tq;
          if (leaf_entry64(l, depth, v, w.tmin[own], w.tmax[own], tq)) key = order_key(tq);
        }
        w.key[lane] = key;
        w.part[lane] = p;
        w.vox[lane] = v;
        __syncwarp();
        const int hi = min(begin + more, base + 32) - base;
        for (int k = max(begin - base, 0); k < hi; ++k) {
          const unsigned long long kk = w.key[k], kv = w.vox[k];
          const uint32_t kp = w.part[k];
          if (kk != kNoHitKey && (kk < best || (kk == best && (kp < part || (kp == part && kv < vox))))) {
            best = kk;
            part = kp;
            vox = kv;
          }
        }
        __syncwarp();
      }
      __syncwarp();  // the entries' local rays are read
      if (nc >= 1) {
        ExactState st;
        st.t = best == kNoHitKey ? Num<double>::inf() : key_value(best);
        st.part = part;
        st.vox = vox;
        write_fixed(L.items[it], ray, st, ((e >> 47) & 1ull) ? SVO_RAY_T_REFINED : SVO_RAY_UNCERTAIN);
      }
      for (unsigned int pending = __ballot_sync(0xffffffffu, have && nc == 0); pending != 0u; pending &= pending - 1u) {
        const int src = __ffs(pending) - 1;
        overflow_retrace(L, i0 + (unsigned long long)src, __shfl_sync(0xffffffffu, e, src), tab,
                         sFix[threadIdx.x >> 5], err, cnt);
      }
    }
  } else
  for (unsigned long long i0 = 4 * warp; i0 < n; i0 += 4 * n_warps) {
    const unsigned long long i = i0 + (unsigned long long)sub;
    const bool have = i < n;
    const unsigned long long e = have ? L.fix_list[i] : 0ull;
    const int nc = (int)(e >> 48);
    {
      // the FP32 pass narrowed the ray to nc contender leaves: lane q of the
      // group takes contenders q and q + 8
      ExactState st;
      st.t = Num<double>::inf();
      st.part = kMissPart;
      st.vox = kMissVoxel;
      const int it = (int)((e >> kRayBits) & 0x7Fu);
      const unsigned long long ray = e & ((1ull << kRayBits) - 1ull);
      if (have && sl < nc) {
        const TraceItem &I = L.items[it];
        const float4 o = I.rays[2 * ray], d = I.rays[2 * ray + 1];
        const uint32_t off = L.fix_off[i];
        for (int q = sl; q < nc; q += 8) {
          const uint4 cv = L.fix_cand[off + q];
          const uint32_t p = cv.x;
          const unsigned long long vox = (unsigned long long)cv.y | ((unsigned long long)cv.z << 32);
          double tq;
          if (leaf_entry64(local_ray64(I.inv64 + 12 * p, o, d), I.aux[p].depth, vox, o.w, d.w, tq)) offer(st, tq, p, vox);
        }
      }
      group_min8(st);
      if (have && nc > 0 && sl == 0)
        write_fixed(L.items[it], ray, st, ((e >> 47) & 1ull) ? SVO_RAY_T_REFINED : SVO_RAY_UNCERTAIN);
    }
    unsigned int pending = __ballot_sync(0xffffffffu, have && nc == 0 && sl == 0);
    while (pending) {
      const int src = __ffs(pending) - 1;
      pending &= pending - 1u;
      const unsigned long long ie = i0 + (unsigned long long)(src >> 3);
      const unsigned long long ee = __shfl_sync(0xffffffffu, e, src);
      overflow_retrace(L, ie, ee, tab, sFix[threadIdx.x >> 5], err, cnt);
    }
  }
  if (L.clean) {
    // Pose changes are tracked relative to a scene's latest trace, and the next
    // trace expects its counters at zero: left so here, by the last block to
    // come through, instead of by memsets around the launches (two per call and
    // one per scene of a batch, each about as long as an empty kernel).
    for (int i = blockIdx.x; i < L.n_items; i += gridDim.x) {
      uint8_t *dirty = const_cast<uint8_t *>(L.items[i].dirty);
      for (int p = threadIdx.x; p < L.items[i].n_parts; p += kBlock) dirty[p] = 0;
    }
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0)  // counts the blocks and wraps to zero with the last
      last = atomicInc(reinterpret_cast<unsigned int *>(&L.clean[kCounterWords - 1]), gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (last)
      for (int k = threadIdx.x; k < (int)kCounterWords - 1; k += kBlock) L.clean[k] = 0ull;
  }
  // count fixed rays once per launch
  if (L.stats && blockIdx.x == 0 && threadIdx.x == 0 && (L.flags & SVO_TRACE_STATS)) atomicAdd(&L.stats->fixed, n);
  if (err) atomicOr(L.err, err);
}

size_t trace_smem_bytes(int stack_levels, int parts, int clusters, int block, int mbox_words, int top_nodes) {
  return kTablesBytes + (size_t)stack_levels * block * sizeof(uint2) + parts * (sizeof(PartHot) + sizeof(PartAux)) +
         clusters * sizeof(Cluster) + (parts + (parts & 1)) * sizeof(int32_t) + (size_t)top_nodes * sizeof(uint2) +
         (size_t)mbox_words * block * sizeof(uint32_t);
}

// Resident blocks per SM of a trace kernel at a dynamic shared-memory size.
// The attribute that admits the size and the occupancy are host calls of a
// few microseconds each, so they are made once per (device, kernel, size); the
// attribute only ever grows, so a size admitted once stays admitted.
struct OccEntry {
  const void *fn;
  int dev;
  size_t smem;
  int per_sm;
};
struct AttrEntry {
  const void *fn;
  int dev;
  size_t smem_max;
};
std::mutex g_occ_mu;
std::vector<OccEntry> g_occ;
std::vector<AttrEntry> g_attr;

template <typename K>
cudaError_t blocks_per_sm(K kern, int block, size_t smem, int &per_sm) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const void *fn = reinterpret_cast<const void *>(kern);
  std::lock_guard<std::mutex> g(g_occ_mu);
  for (const OccEntry &x : g_occ)
    if (x.fn == fn && x.dev == dev && x.smem == smem) {
      per_sm = x.per_sm;
      return cudaSuccess;
    }
  AttrEntry *a = nullptr;
  for (AttrEntry &x : g_attr)
    if (x.fn == fn && x.dev == dev) a = &x;
  if (!a || a->smem_max < smem) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (a)
      a->smem_max = smem;
    else
      g_attr.push_back({fn, dev, smem});
  }
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, block, smem);
  if (e != cudaSuccess) return e;
  g_occ.push_back({fn, dev, smem, per_sm});
  return cudaSuccess;
}

template <int NI, int BLOCK>
cudaError_t launch_trace_b(const TraceLaunchT<NI> &L, const GridLaunch *tile_grids, int n_sm, cudaStream_t stream) {
  const bool stats = (L.flags & SVO_TRACE_STATS) && L.stats;
  const bool reuse = (L.flags & SVO_TRACE_REUSE) != 0;
  bool walk = (L.flags & SVO_TRACE_GRID) != 0 && !reuse;
  if (walk) {
    bool any = false;
    for (int i = 0; i < L.n_items; ++i) any = any || L.items[i].grid != nullptr;
    walk = any;
  }
  if (L.flags & SVO_TRACE_WAVEFRONT) {
    // the culling launch, then the descent launch over the queued rays (the
    // host has checked CULL | SORT without REUSE or GRID)
    const int parts = L.one_scene ? L.items[0].n_parts : 0, clusters = L.one_scene ? L.items[0].n_clusters : 0;
    int max_parts = 0, max_cells = 0;
    for (int i = 0; i < L.n_items; ++i) {
      max_parts = std::max(max_parts, (int)L.items[i].n_parts);
      if (L.items[i].grid && !stats) {
        const int G = grid_cells_per_axis(L.items[i].n_parts);
        max_cells = std::max(max_cells, G * G * G);
      }
    }
    const size_t csmem = cull_smem_bytes(max_parts, max_cells);
    auto ck = stats ? k_cull<NI, true> : k_cull<NI, false>;
    int per_sm = 0;
    cudaError_t e = blocks_per_sm(ck, kCullThreads, csmem, per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    unsigned long long grid = (unsigned long long)n_sm * per_sm;
    const unsigned long long need = (L.n_tiles + kCullWarps - 1) / kCullWarps;
    if (grid > need) grid = need;
    if (grid == 0) return cudaSuccess;
    e = launch_after(ck, (unsigned int)grid, kCullThreads, csmem, stream, L);
    if (e != cudaSuccess) return e;
    // the number of queued rays is known on the device only: a full persistent grid
    const size_t smem = trace_smem_bytes(L.stack_levels, parts, clusters, BLOCK, 0, 0);
    auto kq = stats ? k_descend<NI, true, BLOCK> : k_descend<NI, false, BLOCK>;
    e = blocks_per_sm(kq, BLOCK, smem, per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    e = launch_after(kq, (unsigned int)(n_sm * per_sm), BLOCK, smem, stream, L);
    if constexpr (NI == 1) {
      if (e != cudaSuccess || !L.gate) return e;
      auto kg = k_trace<NI, false, BLOCK, false, false>;
      e = blocks_per_sm(kg, BLOCK, smem, per_sm);
      if (e != cudaSuccess) return e;
      return launch_after(kg, (unsigned int)(n_sm * (per_sm < 1 ? 1 : per_sm)), BLOCK, smem, stream, L);
    }
    return e;
  }
  if (L.tiles) {
    // an image trace: the tile-culling launch, then the trace of the tiles it queued
    int per_sm = 0;
    cudaError_t e = blocks_per_sm(k_tile_cull<NI>, kTileThreads, 0, per_sm);
    if (e != cudaSuccess) return e;
    unsigned long long grid = (unsigned long long)n_sm * (per_sm < 1 ? 1 : per_sm);
    const unsigned long long cull_blocks = (L.n_tiles + kTileThreads / 32 - 1) / (kTileThreads / 32);
    if (grid > cull_blocks) grid = cull_blocks;
    if (grid == 0) return cudaSuccess;
    e = launch_after(k_tile_cull<NI>, (unsigned int)grid, kTileThreads, 0, stream, L);
    if (e != cudaSuccess) return e;
    if (tile_grids) {
      e = launch_grid(*tile_grids, stream);
      if (e != cudaSuccess) return e;
    }
    const size_t smem = trace_smem_bytes(L.stack_levels, L.one_scene ? L.items[0].n_parts : 0,
                                         L.one_scene ? L.items[0].n_clusters : 0, BLOCK, walk ? L.mbox_words : 0, 0);
    auto kl = reuse  ? k_trace<NI, false, BLOCK, true, false, false, true>
              : walk ? k_trace<NI, false, BLOCK, false, true, false, true>
                     : k_trace<NI, false, BLOCK, false, false, false, true>;
    e = blocks_per_sm(kl, BLOCK, smem, per_sm);
    if (e != cudaSuccess) return e;
    grid = (unsigned long long)n_sm * (per_sm < 1 ? 1 : per_sm);
    const unsigned long long blocks = (L.n_tiles + BLOCK / 32 - 1) / (BLOCK / 32);
    if (grid > blocks) grid = blocks;
    return launch_after(kl, (unsigned int)grid, BLOCK, smem, stream, L);
  }
  // the staged top levels only in the common kernel (counting, reuse and grid traces give the same
  // results without them)
  const bool top = L.one_scene && L.top_nodes > 0 && !stats && !reuse && !walk;
  bool image = true;
  for (int i = 0; i < L.n_items; ++i) image = image && L.items[i].tiles_x != 0;
  const size_t smem = trace_smem_bytes(L.stack_levels, L.one_scene ? L.items[0].n_parts : 0,
                                       L.one_scene ? L.items[0].n_clusters : 0, BLOCK, walk ? L.mbox_words : 0,
                                       top ? L.top_nodes : 0);
  auto kern = walk ? (stats ? k_trace<NI, true, BLOCK, false, true> : k_trace<NI, false, BLOCK, false, true>)
              : stats ? (reuse ? k_trace<NI, true, BLOCK, true, false> : k_trace<NI, true, BLOCK, false, false>)
              : reuse ? k_trace<NI, false, BLOCK, true, false>
              : top   ? k_trace<NI, false, BLOCK, false, false, true>
              : image ? k_trace<NI, false, BLOCK, false, false, false, false, true>
                      : k_trace<NI, false, BLOCK, false, false>;
  int per_sm = 0;
  const cudaError_t e = blocks_per_sm(kern, BLOCK, smem, per_sm);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  // one warp per tile: no more blocks than the tiles can keep busy
  unsigned long long grid = (unsigned long long)n_sm * per_sm;
  const unsigned long long need = (L.n_tiles + BLOCK / 32 - 1) / (BLOCK / 32);
  if (grid > need) grid = need;
  if (grid == 0) return cudaSuccess;
  return launch_after(kern, (unsigned int)grid, BLOCK, smem, stream, L);
}

template <int NI>
cudaError_t launch_trace_t(const TraceLaunchT<NI> &L, const GridLaunch *tile_grids, int n_sm, cudaStream_t stream) {
  if (L.block == 64) return launch_trace_b<NI, 64>(L, tile_grids, n_sm, stream);
  if (L.block == 256) return launch_trace_b<NI, 256>(L, tile_grids, n_sm, stream);
  return launch_trace_b<NI, 128>(L, tile_grids, n_sm, stream);
}

// Four blocks, the most that fit: an entry is a chain of dependent reads and
// FP64 instructions, which other warps hide (two blocks: 116 K entries 44 us,
// four 36; re-traces scale with the warps).
constexpr int kFixBlocksPerSM = 4;

template <int NI>
cudaError_t launch_fix_t(const TraceLaunchT<NI> &L, int n_sm, cudaStream_t stream) {
  return launch_after(k_fix<NI>, (unsigned int)(n_sm * kFixBlocksPerSM), kBlock, 0, stream, L);
}

template <int NI>
void fill_launch(const TraceLaunch &src, TraceLaunchT<NI> &dst) {
  for (int i = 0; i < src.n_items && i < NI; ++i) dst.items[i] = src.items[i];
  dst.n_items = src.n_items;
  dst.flags = src.flags;
  dst.n_tiles = src.n_tiles;
  dst.tile_counter = src.tile_counter;
  dst.fix_list = src.fix_list;
  dst.fix_count = src.fix_count;
  dst.fix_capacity = src.fix_capacity;
  dst.fix_cand = src.fix_cand;
  dst.cand_capacity = src.cand_capacity;
  dst.cand_count = src.cand_count;
  dst.fix_off = src.fix_off;
  bool one = true;
  for (int i = 1; i < src.n_items && i < NI; ++i) one = one && src.items[i].hot == src.items[0].hot;
  dst.same_scene = one ? 1 : 0;
  // about four runs per resident block, long enough to repay the staging
  dst.cull_chunk = (int32_t)std::min(128ull, std::max(32ull, src.n_tiles / 2400));
  dst.one_scene = one && src.items[0].n_parts <= kSmemParts ? 1 : 0;
  int lv = 1;
  for (int i = 0; i < src.n_items && i < NI; ++i) lv = src.items[i].max_depth - 1 > lv ? src.items[i].max_depth - 1 : lv;
  dst.stack_levels = lv;
  int mp = 0;
  for (int i = 0; i < src.n_items && i < NI; ++i) mp = src.items[i].n_parts > mp ? src.items[i].n_parts : mp;
  dst.mbox_words = (mp + 31) / 32;
  dst.stats = src.stats;
  dst.err = src.err;
  dst.block = src.block;
  dst.rays_per_lane = src.rays_per_lane < 1 ? 1 : src.rays_per_lane;
  dst.top = src.top;
  dst.top_nodes = (dst.one_scene && src.top) ? src.top_nodes : 0;
  dst.top_levels = dst.top_nodes > 0 ? src.top_levels : 0;
  dst.queue = src.queue;
  dst.queue_count = src.queue_count;
  dst.queue_tile = src.queue_tile;
  dst.tiles = src.tiles;
  dst.tile_count = src.tile_count;
  dst.gate_count = src.gate_count;
  dst.gate = src.gate;
  dst.clean = src.clean;
}

}  // namespace

cudaError_t init_trace_tables(cudaStream_t stream) {
  k_init_tables<<<1, 256, 0, stream>>>();
  return cudaGetLastError();
}

// The kernel parameter block of a batch (about 16 KB): one per host thread,
// allocated on its first batch, so it stays off the caller's stack and off
// the heap of later calls.
TraceLaunchT<kMaxBatchItems> &batch_params() {
  thread_local std::unique_ptr<TraceLaunchT<kMaxBatchItems>> p;
  if (!p) p.reset(new TraceLaunchT<kMaxBatchItems>());
  return *p;
}

cudaError_t launch_trace(const TraceLaunch &L, const GridLaunch *tile_grids, int n_sm, cudaStream_t stream) {
  if (L.n_items <= 1) {
    TraceLaunchT<1> l1;
    fill_launch(L, l1);
    return launch_trace_t(l1, tile_grids, n_sm, stream);
  }
  TraceLaunchT<kMaxBatchItems> &p = batch_params();
  fill_launch(L, p);
  return launch_trace_t(p, tile_grids, n_sm, stream);
}

cudaError_t launch_sample(const TraceLaunch &L, cudaStream_t stream) {
  TraceLaunchT<1> l1;
  fill_launch(L, l1);
  return launch_after(k_sample, kSampleRays / 8, 256, 0, stream, l1);
}

cudaError_t launch_fix(const TraceLaunch &L, int n_sm, cudaStream_t stream) {
  if (L.n_items <= 1) {
    TraceLaunchT<1> l1;
    fill_launch(L, l1);
    return launch_fix_t(l1, n_sm, stream);
  }
  TraceLaunchT<kMaxBatchItems> &p = batch_params();
  fill_launch(L, p);
  return launch_fix_t(p, n_sm, stream);
}

}  // namespace svo
