// k_refit.cu -- per-frame pose pipeline of a scene, one thread block or a
// cluster of up to eight.
//
//  1. compose the transform tree in FP64, parents first: W_i = W_parent(i) o L_i
//     (the paper gives one transform per SVO, Sec. III; the tree is a
//     generalisation in which a root part has W_i = L_i);
//  2. invert each W_i in FP64 (Eq. 3): A^-1 = adj(A)/det(A), b' = -A^-1 b,
//     which for a rigid pose equals the transposed rotation and the negated,
//     rotated translation (Sec. III-A);
//  3. emit the FP32 world->local matrix the trace kernel uses, the local
//     coordinates of the FP32 sphere centre (FP64-accurate), and bounds on
//     norms for the trace kernel's rounding-error bound;
//  4. refit the part bounding spheres (Sec. IV-A: centre and radius follow
//     from the pose).  The sphere bounds the asset's occupied box (the
//     smallest grid-aligned box holding its leaves, found at upload) rather
//     than its whole unit cube: centre = image of the box centre, radius =
//     farthest image of a box corner.  Any sphere that holds every leaf culls
//     no hit; the tighter one culls more rays;
//  5. rebuild the cluster level of the sphere hierarchy: parts sorted by the
//     Morton code of their sphere centres, runs of 8 enclosed by one sphere
//     (the scene-level structure the paper proposes for many parts, Sec. V-E).
//
// GB300 issues FP64 at about two lanes per clock per SM, so one warp's FP64
// instruction occupies a sub-partition for ~64 clocks whatever its active
// lanes.  The kernel therefore (a) spreads the FP64 work of a part over
// three lanes (one matrix row each) and the parts over all eight warps, and
// (b) keeps FP64 for what must be exact -- compose, inverse, sphere centre
// and its local coordinates -- and computes the radii and norms in FP32 with
// upward-rounded error bounds, which only ever enlarge them.
//
// From 65 parts on a scene gets a cluster of blocks, each on an SM of its
// own: one SM's FP64 pipes took 110 of the 153 us of a 1024-part refit.  Every
// block composes the whole tree (roots are copies; a level barrier inside one
// block is cheaper than one across the cluster), inverts and bounds its share
// of the parts, and the blocks exchange spheres, order and clusters through
// global memory between cluster barriers.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include <cfloat>
#include <cmath>
#include <memory>
#include <mutex>

#include "svo_internal.h"

namespace svo {

namespace {

constexpr int kRefitThreads = 256;  // 8 warps: every FP64 sub-partition of the SM gets work
constexpr int kRefitWarps = kRefitThreads / 32;
constexpr int kMaxRefitCluster = 8;  // blocks of a scene's cluster
constexpr int kQuadsPerPass = kRefitThreads / 4;  // parts handled at once (4 lanes each, 3 busy)
constexpr float kRelSlack = 9.5367431640625e-7f;   // 2^-20: covers FP32 rounding of the norms below

// Poses passed by value in the kernel parameters (no host-to-device copy),
// in size classes so that a small scene's launch carries a small parameter
// block (the whole block is fetched before the kernel starts).
template <int CAP>
struct InlinePoses {
  double local[CAP * 12];
};

__device__ __forceinline__ unsigned int spread10(unsigned int v) {
  v &= 0x3FFu;
  v = (v | (v << 16)) & 0x030000FFu;
  v = (v | (v << 8)) & 0x0300F00Fu;
  v = (v | (v << 4)) & 0x030C30C3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

// Thread of the j-th item (part) of a pass.  A warp's FP64 instruction holds
// its sub-partition's FP64 pipe for the same time however few of its lanes
// are busy, so items fill one warp per sub-partition first (warps 0-3, one
// per sub-partition), eight lane groups deep, before warps 4-7 take items 32
// to 63: item j -> warp (j & 3) + 4 (j >> 5), lane group (j >> 2) & 7.  A
// 16-part scene then costs each sub-partition one warp's instructions, not
// two half-empty warps'.  Returns the item handled by thread t and the lane
// r (0..3) inside its group of four.
__device__ __forceinline__ int quad_item(int t, int &r) {
  static_assert(kRefitWarps == 8, "two warps per sub-partition");
  const int w = t >> 5, l = t & 31;
  r = l & 3;
  return 32 * (w >> 2) + 4 * (l >> 2) + (w & 3);
}

// Shared-memory layout of one refit: every per-part intermediate stays on
// chip, so the phases below chain no global-memory round trips (the block
// is alone on its SM and latency-bound).
struct RefitSmem {
  double *world;             // P x 12
  float4 *sph;               // P
  float4 *cl;                // clusters
  unsigned long long *key;   // P
  float *na;                 // P
  int32_t *ord;              // P
  int32_t *parent;           // P
  int32_t *lorder;           // P
  int32_t *lstart;           // levels + 1
  float *red;                // 6 x threads
};

__host__ __device__ inline size_t refit_smem_bytes(int P, int NC, int L, int nthr) {
  return (size_t)P * (12 * sizeof(double) + sizeof(unsigned long long) + sizeof(float4) + sizeof(float) +
                      3 * sizeof(int32_t)) +
         (size_t)NC * sizeof(float4) + (size_t)(L + 1) * sizeof(int32_t) + 6 * (size_t)nthr * sizeof(float) + 64;
}

__device__ inline RefitSmem carve(unsigned char *base, int P, int NC, int L) {
  RefitSmem m;
  // 16-byte items first: every offset stays aligned for any P
  m.world = reinterpret_cast<double *>(base);
  m.sph = reinterpret_cast<float4 *>(m.world + 12 * P);
  m.cl = m.sph + P;
  m.key = reinterpret_cast<unsigned long long *>(m.cl + NC);
  m.na = reinterpret_cast<float *>(m.key + P);
  m.ord = reinterpret_cast<int32_t *>(m.na + P);
  m.parent = m.ord + P;
  m.lorder = m.parent + P;
  m.lstart = m.lorder + P;
  m.red = reinterpret_cast<float *>(m.lstart + L + 1);
  return m;
}

// Upper bound of |x| for x = a - b evaluated in FP32.
__device__ __forceinline__ float abs_diff_up(float a, float b) {
  return fmaxf(fabsf(__fsub_ru(a, b)), fabsf(__fsub_rd(a, b)));
}

// Upper bound of sqrt(x^2 + y^2 + z^2) for non-negative x, y, z.
__device__ __forceinline__ float norm_up(float x, float y, float z) {
  return __fsqrt_ru(__fmaf_ru(x, x, __fmaf_ru(y, y, __fmul_ru(z, z))));
}

// The pose pipeline of one scene.  local: where the local
// poses are read from; keep != nullptr: they are first copied to keep (the
// scene's device copy, kept in step with what is composed), and with
// read_keep the block then reads them back from there (a source in host
// memory is read once).
// The blocks of the launch's cluster (all of them, or one without a cluster
// launch) share the scene's work.
__device__ __forceinline__ void refit_scene(const RefitArgs &a, const double *local, double *keep, bool read_keep,
                                            unsigned char *refit_smem) {
  namespace cg = cooperative_groups;
  wait_for_previous();
  const cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int P = a.n_parts;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int gtid = tid + kRefitThreads * rank, gthreads = kRefitThreads * C;  // in the cluster
  const RefitSmem sm = carve(refit_smem, P, a.n_clusters, a.n_levels);
  // all blocks' global writes before are visible to all after
  const auto sync = [&]() {
    if (C > 1)
      cluster.sync();
    else
      __syncthreads();
  };
  if (keep) {
    for (int k = gtid; k < P * 12; k += gthreads) keep[k] = local[k];
    if (read_keep) {
      local = keep;
      sync();  // the copy below reads what other threads wrote
    }
  }
  // tree topology and local poses to shared memory (independent loads, one
  // round trip: a level below then waits for shared memory only)
  for (int i = tid; i < P; i += kRefitThreads) {
    sm.parent[i] = a.stat[i].parent;
    sm.lorder[i] = a.level_order[i];
  }
  for (int i = tid; i <= a.n_levels; i += kRefitThreads) sm.lstart[i] = a.level_start[i];
#pragma unroll 4
  for (int k = tid; k < P * 12; k += kRefitThreads) sm.world[k] = local[k];
  __syncthreads();

  int r;  // lane inside the part's group of four: rows 0..2, lane 3 helps with the FP32 bounds
  const int q = quad_item(tid, r);
  const unsigned int qmask = 0xFu << (lane & ~3);

  // 1. compose in place, level by level (parents are on earlier levels): a
  //    root's world pose is its local one, and lane r computes row r of
  //    W_i = W_parent o L_i once the group has read all of L_i
  for (int L = 1; L < a.n_levels; ++L) {
    const int b = sm.lstart[L], e = sm.lstart[L + 1];
    for (int j = b + q; j < e; j += kQuadsPerPass) {
      const int i = sm.lorder[j];
      double *Wi = sm.world + 12 * i;
      const double *Wp = sm.world + 12 * sm.parent[i] + 4 * (r < 3 ? r : 2);
      const double p0 = Wp[0], p1 = Wp[1], p2 = Wp[2], p3 = Wp[3];
      double out[4];
      out[0] = p0 * Wi[0] + p1 * Wi[4] + p2 * Wi[8];
      out[1] = p0 * Wi[1] + p1 * Wi[5] + p2 * Wi[9];
      out[2] = p0 * Wi[2] + p1 * Wi[6] + p2 * Wi[10];
      out[3] = p0 * Wi[3] + p1 * Wi[7] + p2 * Wi[11] + p3;
      __syncwarp(qmask);
      if (r < 3) {
#pragma unroll
        for (int c = 0; c < 4; ++c) Wi[4 * r + c] = out[c];
      }
    }
    __syncthreads();
  }
  // change flags against the poses of the previous refit (bitwise; NaN-filled
  // at creation) and the device copy of the world poses, in one pass: one
  // global round trip for the whole scene instead of one per tree level
  for (int k = gtid; k < 12 * P; k += gthreads) {
    const double w = sm.world[k];
    if (__double_as_longlong(a.world[k]) != __double_as_longlong(w)) a.dirty[k / 12] = 1;
    a.world[k] = w;
  }

  // 2-4. per part: lane r < 3 inverts row r in FP64; all four lanes share the
  //      FP32 bounds (radius, norms) through quad shuffles
  float mn[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, mx[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
  const int rr = r < 3 ? r : 2;  // lane 3 repeats row 2 (its FP64 results are not stored)
  for (int p = q + kQuadsPerPass * rank; p < P; p += kQuadsPerPass * C) {
    const double *m = sm.world + 12 * p;
    const double A0 = m[0], A1 = m[1], A2 = m[2], A3 = m[4], A4 = m[5], A5 = m[6], A6 = m[8], A7 = m[9],
                 A8 = m[10];
    const double c00 = A4 * A8 - A5 * A7, c01 = A5 * A6 - A3 * A8, c02 = A3 * A7 - A4 * A6;
    const double det = A0 * c00 + A1 * c01 + A2 * c02;
    // row r of adj(A) = cofactors of column r of A
    const double P1 = rr == 0 ? A2 : (rr == 1 ? A0 : A1), Q1 = rr == 0 ? A7 : (rr == 1 ? A8 : A6);
    const double R1 = rr == 0 ? A1 : (rr == 1 ? A2 : A0), S1 = rr == 0 ? A8 : (rr == 1 ? A6 : A7);
    const double P2 = rr == 0 ? A1 : (rr == 1 ? A2 : A0), Q2 = rr == 0 ? A5 : (rr == 1 ? A3 : A4);
    const double R2 = rr == 0 ? A2 : (rr == 1 ? A0 : A1), S2 = rr == 0 ? A4 : (rr == 1 ? A5 : A3);
    const double e0 = rr == 0 ? c00 : (rr == 1 ? c01 : c02);
    const double e1 = P1 * Q1 - R1 * S1;
    const double e2 = P2 * Q2 - R2 * S2;
    bool ok = isfinite(det) && fabs(det) > 0.0;
    double iv[4] = {0.0, 0.0, 0.0, 0.0};
    if (ok) {
      const double rd = 1.0 / det;
      iv[0] = e0 * rd;
      iv[1] = e1 * rd;
      iv[2] = e2 * rd;
      iv[3] = -(iv[0] * m[3] + iv[1] * m[7] + iv[2] * m[11]);
#pragma unroll
      for (int k = 0; k < 4; ++k) ok = ok && isfinite(iv[k]);
    }
    ok = __all_sync(qmask, ok);
    if (!ok) {
#pragma unroll
      for (int k = 0; k < 4; ++k) iv[k] = 0.0;
      if (r == 0) atomicOr(a.err, kErrSingular);
    }
    if (r < 3) {
#pragma unroll
      for (int k = 0; k < 4; ++k) a.inv64[12 * p + 4 * r + k] = iv[k];
    }
    // sphere centre c = W (lo + hi) / 2 in FP64 (row r), its FP32 rounding,
    // and the local coordinates of that FP32 point (FP64, rounded once)
    const PartStatic &ps = a.stat[p];
    const float lo0 = ps.box_lo[0], lo1 = ps.box_lo[1], lo2 = ps.box_lo[2];
    const float hi0 = ps.box_hi[0], hi1 = ps.box_hi[1], hi2 = ps.box_hi[2];
    const double mid0 = 0.5 * ((double)lo0 + (double)hi0), mid1 = 0.5 * ((double)lo1 + (double)hi1),
                 mid2 = 0.5 * ((double)lo2 + (double)hi2);
    const double cr = m[4 * rr] * mid0 + m[4 * rr + 1] * mid1 + m[4 * rr + 2] * mid2 + m[4 * rr + 3];
    const float cfr = (float)cr;
    const float cfx = __shfl_sync(qmask, cfr, 0, 4), cfy = __shfl_sync(qmask, cfr, 1, 4),
                cfz = __shfl_sync(qmask, cfr, 2, 4);
    const float lcr = (float)(iv[0] * (double)cfx + iv[1] * (double)cfy + iv[2] * (double)cfz + iv[3]);
    const float f0 = (float)iv[0], f1 = (float)iv[1], f2 = (float)iv[2];
    if (r < 3) reinterpret_cast<float4 *>(&a.hot[p])[r] = make_float4(f0, f1, f2, lcr);
    // FP32 bounds, every sum of squares rounded up.  Box half extents and
    // the corner offsets +-e are exact in FP32 (multiples of 2^-depth).
    const bool row = r < 3;
    float rs = row ? __fadd_ru(__fadd_ru(fabsf(f0), fabsf(f1)), fabsf(f2)) : 0.f;  // row of |Ainv|
    const float ex0 = 0.5f * (hi0 - lo0), ex1 = 0.5f * (hi1 - lo1), ex2 = 0.5f * (hi2 - lo2);
    const float a0 = (float)m[4 * rr], a1 = (float)m[4 * rr + 1], a2 = (float)m[4 * rr + 2];
    const float u0 = a0 * ex0, u1 = a1 * ex1, u2 = a2 * ex2;
    float s[7];
    s[0] = u0 + u1 + u2;  // the four corner directions (the other four are their negatives)
    s[1] = u0 + u1 - u2;
    s[2] = u0 - u1 + u2;
    s[3] = u0 - u1 - u2;
    s[4] = fabsf(u0) + fabsf(u1) + fabsf(u2);  // |A| e: scale of every rounding error above
    s[5] = a0 + a1 + a2;                          // A (1,1,1): the leaf diagonal direction
    s[6] = (float)fabs(cr - (double)cfr);         // centre rounding
#pragma unroll
    for (int k = 0; k < 7; ++k) {
      float v = row ? __fmul_ru(s[k], s[k]) : 0.f;
      v = __fadd_ru(v, __shfl_xor_sync(qmask, v, 1, 4));
      v = __fadd_ru(v, __shfl_xor_sync(qmask, v, 2, 4));
      s[k] = v;
    }
    rs = fmaxf(rs, __shfl_xor_sync(qmask, rs, 1, 4));
    rs = fmaxf(rs, __shfl_xor_sync(qmask, rs, 2, 4));
    if (r == 0) {
      // |A q - c| <= computed + rounding (<= 2^-20 |A| e) for every corner q,
      // plus the distance of the FP32 centre from the exact one
      const float rfl = __fsqrt_ru(fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3])));
      const float rad = __fadd_ru(__fadd_ru(__fmul_ru(rfl, 1.0f + kRelSlack), __fmul_ru(__fsqrt_ru(s[4]), kRelSlack)),
                                  __fmul_ru(__fsqrt_ru(s[6]), 1.0f + kRelSlack));
      // a singular pose or an empty asset disables the sphere: no ray tests the part
      const float4 sph = make_float4(cfx, cfy, cfz, (ok && ps.n_nodes > 0) ? rad : -1.0f);
      reinterpret_cast<float4 *>(&a.hot[p])[3] = sph;
      sm.sph[p] = sph;
      a.sphere[p] = sph;
      PartAux x;
      x.nodes = ps.nodes;
      x.n_nodes = ps.n_nodes;
      x.depth = ps.depth;
      x.n_ainv = rs;
      x.hdiag = sqrtf(s[5]) * __int_as_float((127 - ps.depth) << 23);
      x.spare0 = 0.f;
      x.spare1 = 0.f;
      for (int k = 0; k < 3; ++k) {
        x.box_lo[k] = ps.box_lo[k];
        x.box_hi[k] = ps.box_hi[k];
      }
      x.pad[0] = x.pad[1] = 0.f;
      a.aux[p] = x;
      sm.na[p] = rs;
      mn[0] = fminf(mn[0], cfx);
      mn[1] = fminf(mn[1], cfy);
      mn[2] = fminf(mn[2], cfz);
      mx[0] = fmaxf(mx[0], cfx);
      mx[1] = fmaxf(mx[1], cfy);
      mx[2] = fmaxf(mx[2], cfz);
    }
  }
  // bounding box of the sphere centres: warp shuffles, then the warps'
  // results of every block (min and max are exact in any order)
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mn[k] = fminf(mn[k], __shfl_xor_sync(0xffffffffu, mn[k], o));
      mx[k] = fmaxf(mx[k], __shfl_xor_sync(0xffffffffu, mx[k], o));
    }
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      sm.red[k * kRefitWarps + (tid >> 5)] = mn[k];
      sm.red[(3 + k) * kRefitWarps + (tid >> 5)] = mx[k];
    }
  }
  sync();
  float bb[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) bb[k] = k < 3 ? FLT_MAX : -FLT_MAX;
  for (int b = 0; b < C; ++b) {
    const float *red = C > 1 ? cluster.map_shared_rank(sm.red, b) : sm.red;
#pragma unroll
    for (int k = 0; k < 6; ++k)
      for (int w = 0; w < kRefitWarps; ++w)
        bb[k] = k < 3 ? fminf(bb[k], red[k * kRefitWarps + w]) : fmaxf(bb[k], red[k * kRefitWarps + w]);
  }
  if (C > 1)  // the other blocks' spheres
    for (int i = tid; i < P; i += kRefitThreads) sm.sph[i] = a.sphere[i];
  const float bx0 = bb[0], by0 = bb[1], bz0 = bb[2];
  const float bx1 = bb[3], by1 = bb[4], bz1 = bb[5];
  const float ex = fmaxf(bx1 - bx0, 1e-30f), ey = fmaxf(by1 - by0, 1e-30f), ez = fmaxf(bz1 - bz0, 1e-30f);
  // 5. Morton keys and a rank sort (P <= kMaxParts)
  for (int i = tid; i < P; i += kRefitThreads) {  // thread i holds sphere i
    const float4 s = sm.sph[i];
    const unsigned int qx = (unsigned int)fminf(fmaxf((s.x - bx0) / ex * 1023.0f, 0.0f), 1023.0f);
    const unsigned int qy = (unsigned int)fminf(fmaxf((s.y - by0) / ey * 1023.0f, 0.0f), 1023.0f);
    const unsigned int qz = (unsigned int)fminf(fmaxf((s.z - bz0) / ez * 1023.0f, 0.0f), 1023.0f);
    const unsigned int mc = spread10(qx) | (spread10(qy) << 1) | (spread10(qz) << 2);
    sm.key[i] = ((unsigned long long)mc << 11) | (unsigned long long)i;
  }
  __syncthreads();
  // a part's rank by `per` neighbouring threads, each against its share of the keys
  int per = 1;
  while (per < 8 && 2 * per * P <= gthreads) per *= 2;
  for (int w = gtid - lane; w < P * per; w += gthreads) {  // whole warps: the shuffles below need them
    const int i = (w + lane) / per, part = (w + lane) % per;
    const unsigned long long k = i < P ? sm.key[i] : 0ull;
    int pos = 0;
    for (int j = part; j < P; j += per) pos += (sm.key[j] < k) ? 1 : 0;
    for (int o = 1; o < per; o <<= 1) pos += __shfl_xor_sync(0xffffffffu, pos, o);
    if (i < P && part == 0) {
      sm.ord[pos] = i;
      a.order[pos] = i;
      a.sph[pos] = sm.sph[i];
    }
  }
  sync();
  // clusters: a sphere around the member spheres, in FP32 rounded outward;
  // eight lanes each, one a member
  static_assert(kClusterSize == 8, "eight lanes a cluster");
  for (int w = gtid - lane; w < a.n_clusters * kClusterSize; w += gthreads) {
    const int cidx = (w + lane) >> 3, k = lane & 7;
    const int first = cidx * kClusterSize;
    const int cnt = min(kClusterSize, P - first);  // not positive past the last cluster
    const int p = k < cnt ? (C > 1 ? a.order[first + k] : sm.ord[first + k]) : -1;
    const float4 s = p >= 0 ? sm.sph[p] : make_float4(0.f, 0.f, 0.f, -1.0f);
    const bool in = p >= 0 && !(s.w < 0.f);
    float lo[3], hi[3];
    lo[0] = in ? __fsub_rd(s.x, s.w) : FLT_MAX;
    lo[1] = in ? __fsub_rd(s.y, s.w) : FLT_MAX;
    lo[2] = in ? __fsub_rd(s.z, s.w) : FLT_MAX;
    hi[0] = in ? __fadd_ru(s.x, s.w) : -FLT_MAX;
    hi[1] = in ? __fadd_ru(s.y, s.w) : -FLT_MAX;
    hi[2] = in ? __fadd_ru(s.z, s.w) : -FLT_MAX;
    float na = in ? (C > 1 ? a.aux[p].n_ainv : sm.na[p]) : 0.f;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
        hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
      }
      na = fmaxf(na, __shfl_xor_sync(0xffffffffu, na, o));
    }
    const bool any = hi[0] >= lo[0];
    // any centre works: the radius is measured from it with upward rounding
    const float Cx = 0.5f * lo[0] + 0.5f * hi[0], Cy = 0.5f * lo[1] + 0.5f * hi[1], Cz = 0.5f * lo[2] + 0.5f * hi[2];
    float R = in ? __fadd_ru(norm_up(abs_diff_up(s.x, Cx), abs_diff_up(s.y, Cy), abs_diff_up(s.z, Cz)), s.w) : 0.f;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) R = fmaxf(R, __shfl_xor_sync(0xffffffffu, R, o));
    if (k == 0 && cidx < a.n_clusters) {
      Cluster cl;
      cl.sphere = any ? make_float4(Cx, Cy, Cz, R) : make_float4(0.f, 0.f, 0.f, -1.0f);
      cl.aux = make_float4(na, 0.f, 0.f, __uint_as_float((unsigned int)first | ((unsigned int)cnt << 16)));
      a.clusters[cidx] = cl;
      sm.cl[cidx] = cl.sphere;
    }
  }
  sync();
  if (rank == 0 && tid < 32) {
    // a sphere around all cluster spheres: the frame of origin-based ray ordering
    const float Cx = 0.5f * (bx0 + bx1), Cy = 0.5f * (by0 + by1), Cz = 0.5f * (bz0 + bz1);
    float R = 0.f;
    for (int c = lane; c < a.n_clusters; c += 32) {
      const float4 s = C > 1 ? a.clusters[c].sphere : sm.cl[c];
      if (s.w < 0.f) continue;
      R = fmaxf(R, __fadd_ru(norm_up(abs_diff_up(s.x, Cx), abs_diff_up(s.y, Cy), abs_diff_up(s.z, Cz)), s.w));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) R = fmaxf(R, __shfl_xor_sync(0xffffffffu, R, o));
    if (lane == 0) *a.bound = make_float4(Cx, Cy, Cz, R);
  }
  // the scene grid, if any, no longer matches the spheres: the next grid
  // trace rebuilds it first
  if (a.grid != nullptr && gtid == 0) a.grid->stale = kGridStale;
}

template <bool INLINE, int CAP>
__global__ void __launch_bounds__(kRefitThreads) k_refit(RefitArgs a, const __grid_constant__ InlinePoses<CAP> poses) {
  extern __shared__ __align__(16) unsigned char refit_smem[];
  // inline poses: composed from the parameter block, and copied to the
  // scene's device copy on the way
  refit_scene(a, INLINE ? poses.local : a.local, INLINE ? const_cast<double *>(a.local) : nullptr, false, refit_smem);
}

// Many scenes in one launch, one cluster of blocks each (scene_refit_batch):
// cluster b refits B.a[b], reading its local poses from B.src[b] (device or mapped
// host memory) when that is set.
struct RefitBatch {
  RefitArgs a[kRefitBatch];
  const double *src[kRefitBatch];
  int32_t n;
  int32_t cluster;  // blocks a scene
};

__global__ void __launch_bounds__(kRefitThreads) k_refit_batch(const __grid_constant__ RefitBatch B) {
  extern __shared__ __align__(16) unsigned char refit_smem[];
  const int b = blockIdx.x / B.cluster;
  const RefitArgs &a = B.a[b];
  const double *src = B.src[b];
  refit_scene(a, src ? src : a.local, src ? const_cast<double *>(a.local) : nullptr, true, refit_smem);
}

// Blocks of a scene's cluster: a block takes 64 parts a pass, two warps on
// each FP64 pipe.  Measured per refit, one block (of the code before) against
// the cluster: 1024 parts 153 -> 52 us (4 blocks: 72), 128 parts 25.6 -> 19.1,
// 64 scenes of up to 256 parts in one launch 42 -> 27 (32 parts a block: 53,
// the launch then waits for room for its clusters).
//
// Many large scenes in one launch get smaller clusters, so that every block has
// an SM to itself: two blocks on one SM share its FP64 pipes, and clusters that
// find no room wait for a whole round.  n_full: the scenes the launch would hold
// if all were as large as its largest.  Per launch, clusters of 1 / 2 / 4 / 8:
//   1024 parts, 12 scenes 425 / 315 / 260 / 240 us, 16: 426 / 316 / 259 / 465,
//               64: 432 / 320 / 517 / 1158
//   512 parts,  12 scenes 198 / 159 / 139 / 138,    32: 198 / 158 / 140 / 183,
//               64: 200 / 160 / 184 / 358
//   256 parts,  32 scenes  93 /  79 /  72 / 109,    64:  94 /  80 / 100 / 165
int refit_cluster(int n_parts, int n_full) {
  int c = 1;
  while (c < kMaxRefitCluster && 64 * c < n_parts) c *= 2;
  while (c > 2 && n_full > (c > 4 ? 12 : 32)) c /= 2;
  return c;
}

template <typename... Params, typename... Args>
cudaError_t launch_clusters(void (*kern)(Params...), int n, int cluster, size_t smem, cudaStream_t stream,
                            const Args &...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned int)(n * cluster));
  cfg.blockDim = dim3(kRefitThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned int)cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <bool INLINE, int CAP>
cudaError_t launch_refit_t(const RefitArgs &a, const double *host_local, size_t smem, cudaStream_t stream) {
  InlinePoses<CAP> p;
  if (INLINE)
    for (int k = 0; k < a.n_parts * 12; ++k) p.local[k] = host_local[k];
  cudaError_t e = cudaFuncSetAttribute(k_refit<INLINE, CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_clusters(k_refit<INLINE, CAP>, 1, refit_cluster(a.n_parts, 1), smem, stream, a, p);
}

}  // namespace

cudaError_t launch_refit_batch(const RefitArgs *args, const double *const *src, int n, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  if (n > kRefitBatch) return cudaErrorInvalidValue;
  // the parameter block (about 9 KB): one per host thread, allocated on its
  // first batched refit, so it stays off the caller's stack and no call
  // allocates it afresh
  thread_local std::unique_ptr<RefitBatch> block;
  if (!block) block.reset(new RefitBatch());
  RefitBatch &B = *block;
  size_t smem = 0;
  for (int i = 0; i < n; ++i) {
    B.a[i] = args[i];
    B.src[i] = src[i];
    const size_t m = refit_smem_bytes(args[i].n_parts, args[i].n_clusters, args[i].n_levels, kRefitThreads);
    smem = m > smem ? m : smem;
  }
  B.n = n;
  int parts = 1, total = 0;
  for (int i = 0; i < n; ++i) {
    parts = std::max(parts, (int)args[i].n_parts);
    total += args[i].n_parts;
  }
  B.cluster = refit_cluster(parts, (total + parts - 1) / parts);
  // the shared-memory attribute only ever grows: set it when this launch needs more (per device)
  constexpr int kMaxDevices = 64;
  static std::mutex mu;
  static size_t admitted[kMaxDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  {
    std::lock_guard<std::mutex> g(mu);
    if (smem > admitted[dev]) {
      e = cudaFuncSetAttribute(k_refit_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      admitted[dev] = smem;
    }
  }
  return launch_clusters(k_refit_batch, n, B.cluster, smem, stream, B);
}

cudaError_t launch_refit(const RefitArgs &a, const double *host_local, cudaStream_t stream) {
  static_assert(kInlinePoseParts == 256, "size classes below");
  const size_t smem = refit_smem_bytes(a.n_parts, a.n_clusters, a.n_levels, kRefitThreads);
  if (host_local && a.n_parts <= 16) return launch_refit_t<true, 16>(a, host_local, smem, stream);
  if (host_local && a.n_parts <= 64) return launch_refit_t<true, 64>(a, host_local, smem, stream);
  if (host_local && a.n_parts <= 256) return launch_refit_t<true, 256>(a, host_local, smem, stream);
  return launch_refit_t<false, 1>(a, nullptr, smem, stream);
}

}  // namespace svo
