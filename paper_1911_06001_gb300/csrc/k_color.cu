// k_color.cu -- what shading needs of the closest hits.
//
// The hit buffer of the paper (Sec. IV-C) carries, per pixel, the closest
// hit's colour and normal for shading.  For a voxel model:
//   * colour: the hit leaf's payload.  A hit (part, voxel id) is resolved to
//     its leaf by walking the part's octree from the root along the voxel's
//     coordinate bits: at level l the child octant is bit D-1-l of x, y and z
//     (bit 0 of the octant = +x); the leaf-level node's first_child indexes
//     the leaf payload array directly;
//   * normal: the face of the leaf's box through which the ray enters, mapped
//     to world space by the inverse transpose of the part's pose (so that
//     shear and anisotropic scale keep it perpendicular to the face).
// trace_shade combines both into a Lambert-lit 8-bit image.  Its decisions
// (entry face, rounding of each channel) are those of FP64, like the FP64
// re-intersection pass, so that they match an FP64 evaluation of the same
// rule except within rounding distance of a tie: FP32 takes those that its
// error bounds settle (shade_fast), FP64 the rest (shade_exact).
#include <cuda_runtime.h>

#include <cstdint>

#include "svo_internal.h"

namespace svo {

namespace {

// Payload of the leaf (part, vox) names, SVO_COLOR_INVALID if it names none.
__device__ __forceinline__ uint32_t leaf_color(const PartStatic &ps, unsigned long long vox) {
  const int D = ps.depth;
  const unsigned long long mask = (1ull << D) - 1ull;
  if (ps.n_nodes == 0 || (vox >> (3 * D)) != 0ull) return SVO_COLOR_INVALID;
  const uint32_t x = (uint32_t)(vox & mask), y = (uint32_t)((vox >> D) & mask), z = (uint32_t)((vox >> (2 * D)) & mask);
  uint32_t node = 0;
  for (int l = 0; l < D; ++l) {
    const int b = D - 1 - l;
    const uint32_t k = ((x >> b) & 1u) | (((y >> b) & 1u) << 1) | (((z >> b) & 1u) << 2);
    const uint2 d = __ldg(&ps.nodes[node]);
    const uint32_t cmask = d.y & 0xFFu;
    if (!((cmask >> k) & 1u)) return SVO_COLOR_INVALID;  // not occupied
    const uint32_t idx = d.x + __popc(cmask & ((1u << k) - 1u));
    if (l == D - 1) return idx < ps.n_leaves ? __ldg(&ps.rgb[idx]) : SVO_COLOR_INVALID;
    if (idx >= ps.n_nodes) return SVO_COLOR_INVALID;
    node = idx;
  }
  return SVO_COLOR_INVALID;
}

__device__ __forceinline__ uint32_t hit_color(const uint4 h, const PartStatic *__restrict__ stat, int n_parts,
                                              uint32_t background) {
  if (h.y == kMissPart) return background;
  if (h.y >= (uint32_t)n_parts) return SVO_COLOR_INVALID;
  return leaf_color(stat[h.y], ((unsigned long long)h.w << 32) | h.z);
}

__global__ void k_hit_colors(const uint4 *__restrict__ hits, unsigned long long n,
                             const PartStatic *__restrict__ stat, int n_parts, uint32_t background,
                             uint32_t *__restrict__ rgb) {
  wait_for_previous();
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    __stcs(&rgb[i], hit_color(__ldcs(&hits[i]), stat, n_parts, background));
}

// One 8-bit channel scaled by s and rounded half up, at most 255.
__device__ __forceinline__ uint32_t shade_channel(uint32_t c, double s) {
  const double x = floor((double)c * s + 0.5);
  return x >= 255.0 ? 255u : (uint32_t)x;
}

// The shaded colour of one hit, decided in FP64.
__device__ __noinline__ uint32_t shade_exact(uint32_t color, float4 o, float4 d, const double *__restrict__ m, int D,
                                             unsigned long long vox, const ShadeArgs &sa) {
  const unsigned long long mask = (1ull << D) - 1ull;
  const double size = __longlong_as_double((long long)(1023 - D) << 52);  // 2^-D
  const double ro[3] = {o.x, o.y, o.z}, rd[3] = {d.x, d.y, d.z};
  // entry face: the axis whose near-plane t is largest (lower axis on a tie)
  double te = -__longlong_as_double(0x7ff0000000000000ll);
  int kf = 0;
  double sgn = 0.0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double ol = m[4 * k] * ro[0] + m[4 * k + 1] * ro[1] + m[4 * k + 2] * ro[2] + m[4 * k + 3];
    const double dl = m[4 * k] * rd[0] + m[4 * k + 1] * rd[1] + m[4 * k + 2] * rd[2];
    if (dl == 0.0) continue;
    const double lo = (double)((vox >> (k * D)) & mask) * size;
    const double t = ((dl > 0.0 ? lo : lo + size) - ol) / dl;
    if (t > te) {
      te = t;
      kf = k;
      sgn = dl > 0.0 ? 1.0 : -1.0;
    }
  }
  double nx, ny, nz;
  if (te < (double)o.w || sgn == 0.0) {  // the ray starts inside the leaf: face the viewer
    nx = -rd[0];
    ny = -rd[1];
    nz = -rd[2];
  } else {  // outward face normal -sign(d'_k) e_k, through the inverse transpose
    nx = -sgn * m[4 * kf];
    ny = -sgn * m[4 * kf + 1];
    nz = -sgn * m[4 * kf + 2];
  }
  const double len = sqrt(nx * nx + ny * ny + nz * nz);
  const double cosl = (nx * sa.light[0] + ny * sa.light[1] + nz * sa.light[2]) / len;
  const double s = sa.ambient + (1.0 - sa.ambient) * (cosl > 0.0 ? cosl : 0.0);
  return (shade_channel((color >> 16) & 255u, s) << 16) | (shade_channel((color >> 8) & 255u, s) << 8) |
         shade_channel(color & 255u, s);
}

// One 8-bit channel scaled by s, known to within 1e-6, and rounded half up;
// sure: cleared where that error could change the result (255 x 1e-6 and the
// roundings here, from a half; 4e-4 covers both).
__device__ __forceinline__ uint32_t shade_channel_fast(uint32_t c, float s, bool &sure) {
  const float x = fmaf((float)c, s, 0.5f), f = floorf(x), r = x - f;
  sure = sure && r > 4e-4f && r < 1.0f - 4e-4f;
  return f >= 255.f ? 255u : (uint32_t)f;
}

// An upper bound of |x| in FP32 from its high word (FP64 instructions are what
// bounds this kernel), clamped to [2^-126, 2^127]: the bounds below are then
// decided by their other terms, or fail.
__device__ __forceinline__ float mag_up(double x) {
  const int h = min(max(__double2hiint(x) & 0x7fffffff, 897 << 20), (1150 << 20) - 1);
  return __int_as_float((h - (896 << 20) + 1) << 3);
}

// The same decisions taken in FP32 wherever their error cannot change them.
// The ray is moved to its hit's t in FP64, so that what FP32 compares are the
// distances from the leaf's planes, leaves in size: u_k with an error of 2^-24
// of (|u_k| + size), tau_k = u_k / d'_k within e_k below.  To that comes the FP64
// rounding of both ways: of the origin's transform, a chain of up to five
// operations on terms of at most mo that may cancel (a part far from the world's
// origin, a small part), 5 + 3 units of 2^-53 mo, and of the direction's, 4 + 3
// units of md for each t moved along it.  Where eleven units of them (1.2e-15) are
// more than 2^-24 of (|u_k| + size) the exact way is taken.  n_ainv: the inverse's
// infinity norm, rounded up.  Returns false there, and where the entry face, the
// test for a start inside the leaf or a channel's rounding is too close to call.
__device__ __forceinline__ bool shade_fast(uint32_t color, float t, float4 o, float4 d, const double *__restrict__ m,
                                           float n_ainv, int D, unsigned long long vox, const ShadeArgs &sa,
                                           uint32_t &out) {
  constexpr float kU32 = 5.9604644775390625e-8f;  // 2^-24
  const uint32_t mask = (1u << D) - 1u;
  const double size64 = __longlong_as_double((long long)(1023 - D) << 52);
  const float size = __int_as_float((127 - D) << 23);
  const float md = n_ainv * fmaxf(fmaxf(fabsf(d.x), fabsf(d.y)), fabsf(d.z));
  const float mo = fmaf(n_ainv, fmaxf(fmaxf(fabsf(o.x), fabsf(o.y)), fabsf(o.z)),
                        fmaxf(fmaxf(mag_up(m[3]), mag_up(m[7])), mag_up(m[11])));
  if (!(1.2e-15f * (2.0f + fmaf(fabsf(t), md, mo)) <= kU32 * size)) return false;
  const float dmin = fmaxf(1e-20f, 2.1e-8f * md);  // 1.2e-15 |tau| md <= 2^-24 |u| from here on
  const double ox = o.x, oy = o.y, oz = o.z, dx = d.x, dy = d.y, dz = d.z, th = t;
  float best = -__int_as_float(0x7f800000), err = 0.f, next = best, next_err = 0.f;
  int kf = -1;
  bool back = false, sure = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double ol = fma(m[4 * k], ox, fma(m[4 * k + 1], oy, fma(m[4 * k + 2], oz, m[4 * k + 3])));
    const double dl = fma(m[4 * k], dx, fma(m[4 * k + 1], dy, m[4 * k + 2] * dz));
    const double lo = (double)((uint32_t)(vox >> (k * D)) & mask) * size64;
    const float u0 = (float)(lo - fma(th, dl, ol)), dk = (float)dl;
    const float u = dk > 0.f ? u0 : u0 + size;
    const float inv = __frcp_rn(dk);
    const float tau = u * inv, e = 10.0f * kU32 * (fabsf(u) + size) * fabsf(inv);
    sure = sure && fabsf(dk) > dmin && fabsf(dk) < 1e20f;  // a zero or extreme component: the exact way
    if (tau > best) {
      if (best + err > next + next_err) {
        next = best;
        next_err = err;
      }
      best = tau;
      err = e;
      kf = k;
      back = dk < 0.f;
    } else if (tau + e > next + next_err) {
      next = tau;
      next_err = e;
    }
  }
  sure = sure && best - err > next + next_err;
  // entered from outside, beyond the rounding of t and tmin (te < tmin: inside)
  const float te = t + best;
  sure = sure && te - o.w > 4.0f * kU32 * (fabsf(t) + fabsf(te) + fabsf(o.w)) + err;
  if (!sure) return false;
  const double *row = m + 4 * kf;
  const float nx = (float)row[0], ny = (float)row[1], nz = (float)row[2];
  const float dot = nx * (float)sa.light[0] + ny * (float)sa.light[1] + nz * (float)sa.light[2];
  const float n2 = nx * nx + ny * ny + nz * nz;
  sure = n2 > 1e-30f && n2 < 1e30f;
  // |cos| within 8 x 2^-24 of its value: the light is a unit vector
  const float cosl = (back ? dot : -dot) * rsqrtf(n2);
  const float amb = (float)sa.ambient;
  const float s = fmaf(1.0f - amb, fmaxf(cosl, 0.f), amb);
  out = (shade_channel_fast((color >> 16) & 255u, s, sure) << 16) |
        (shade_channel_fast((color >> 8) & 255u, s, sure) << 8) | shade_channel_fast(color & 255u, s, sure);
  return sure;
}

// One thread per pixel.  Bound by the FP64 pipes: with every decision in FP64
// (two matrix products, three divisions, a square root and a channel each
// about seven instructions) 0.16 M hits of 0.98 M pixels took 57 us, now 28.
__global__ void k_shade(const float4 *__restrict__ rays, const uint4 *__restrict__ hits, unsigned long long n,
                        const PartStatic *__restrict__ stat, const PartAux *__restrict__ aux,
                        const double *__restrict__ inv64, int n_parts, const __grid_constant__ ShadeArgs sa, uint32_t *__restrict__ rgb) {
  wait_for_previous();
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const uint4 h = __ldcs(&hits[i]);
    uint32_t out = hit_color(h, stat, n_parts, sa.background);
    if (h.y != kMissPart && out != SVO_COLOR_INVALID) {
      const float4 o = __ldcs(&rays[2 * i]), d = __ldcs(&rays[2 * i + 1]);
      const double *m = inv64 + 12 * (size_t)h.y;
      const unsigned long long vox = ((unsigned long long)h.w << 32) | h.z;
      const int D = stat[h.y].depth;
      uint32_t lit;
      if (!shade_fast(out, __uint_as_float(h.x), o, d, m, aux[h.y].n_ainv, D, vox, sa, lit))
        lit = shade_exact(out, o, d, m, D, vox, sa);
      out = lit;
    }
    __stcs(&rgb[i], out);
  }
}

unsigned int grid_for(unsigned long long n, int threads, int n_sm) {
  const unsigned long long want = (n + threads - 1) / threads;
  const unsigned long long cap = (unsigned long long)n_sm * 8ull;  // 8 resident blocks per SM
  return (unsigned int)(want < cap ? want : cap);
}

}  // namespace

cudaError_t launch_hit_colors(const uint4 *hits, unsigned long long n, const PartStatic *stat, int n_parts,
                              uint32_t background, uint32_t *rgb, int n_sm, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  return launch_after(k_hit_colors, grid_for(n, 256, n_sm), 256, 0, stream, hits, n, stat, n_parts, background, rgb);
}

cudaError_t launch_shade(const float4 *rays, const uint4 *hits, unsigned long long n, const PartStatic *stat,
                         const PartAux *aux, const double *inv64, int n_parts, const ShadeArgs &sa, uint32_t *rgb, int n_sm,
                         cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  return launch_after(k_shade, grid_for(n, 256, n_sm), 256, 0, stream, rays, hits, n, stat, aux, inv64, n_parts, sa, rgb);
}

}  // namespace svo
