// vd_walk.cuh -- culling tests and FP64 helpers shared by the kernels that
// walk the 8-wide tree (vd_quad.cu, four cells per warp; vd_solo.cu, one).
#pragma once

#include "vd_clip.cuh"

namespace vd {

// sqrt to a few units in the last place: the culling bounds it feeds are
// padded by 1e-5
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Bounds of a cell for the culling tests: its vertex box and the squares of
// its sides, its bounding sphere, the square of that sphere's farthest point
// from the site, and a length that bounds every coordinate involved.
struct WalkBounds {
  float lo[3], hi[3], lo2[3], hi2[3], c[3], rad, reach2, ext;
};

// Candidate test of Sec. 4.2.1 (candidate_test in vd_clip.cuh, one padding
// term for both halves): may the plane n.x <= beta cut the box and the
// sphere? No branches: every lane of the warp has a site to test.
__device__ __forceinline__ bool walk_site_test(float nx, float ny, float nz, float nn, float wi, float wj,
                                               const WalkBounds& B) {
  const float beta = 0.5f * (nn + (wi - wj));
  const float slack = kCullPad * fmaf(fabsf(nx) + fabsf(ny) + fabsf(nz), B.ext, nn + fabsf(wi) + fabsf(wj));
  const float sup = fmaxf(nx * B.lo[0], nx * B.hi[0]) + fmaxf(ny * B.lo[1], ny * B.hi[1]) +
                    fmaxf(nz * B.lo[2], nz * B.hi[2]);
  const float rhs = beta - slack - fmaf(nx, B.c[0], fmaf(ny, B.c[1], nz * B.c[2]));
  return (sup > beta - slack) & ((rhs <= 0.f) | (B.rad * B.rad * nn > rhs * rhs));
}

// Node test of Sec. 4.2.2 (see node_test_r in vd_clip.cuh for the bound):
// may a site of the box [lo, hi] (maximum weight lo.w) cut the cell? `key`
// orders the nodes, best first; `lb` is a lower bound of the sites' d_ij. The squared radius over the octants that
// the box occupies is formed without building the octant mask, and without
// weights the bound D / 2 > R is tested on squares (the same test up to its
// padding).
__device__ __forceinline__ bool walk_node_test(const float4 lo, const float4 hi, const float4 me, const WalkBounds& B,
                                               bool weighted, float& key, float& lb) {
  const float rl[3] = {lo.x - me.x, lo.y - me.y, lo.z - me.z};
  const float rh[3] = {hi.x - me.x, hi.y - me.y, hi.z - me.z};
  float d2 = 0.f, r2 = 0.f;
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const float d = fmaxf(fmaxf(rl[k], -rh[k]), 0.f);
    d2 = fmaf(d, d, d2);
    r2 += fmaxf(rh[k] >= 0.f ? B.hi2[k] : 0.f, rl[k] <= 0.f ? B.lo2[k] : 0.f);
  }
  r2 = fminf(r2, B.reach2);
  const float R = sqrt_approx(r2);
  float D = sqrt_approx(d2);
  if (!weighted) {
    key = fmaf(0.5f, D, -R);
    lb = D * (0.5f * (1.0f - 2.0f * kCullPad));
    return !(d2 > r2 * (4.0f * (1.0f + 10.0f * kCullPad)));
  }
  const float c = me.w - lo.w;
  if (c > 0.f) {
    float f2 = 0.f;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const float f = fmaxf(fabsf(rl[k]), fabsf(rh[k]));
      f2 = fmaf(f, f, f2);
    }
    D = fminf(fmaxf(sqrt_approx(c), D), sqrt_approx(f2) * (1.0f + kCullPad));
  }
  key = -R;
  lb = -INFINITY;
  if (!(D > 0.f)) return true;
  const float D2 = D * D, inv = __fdividef(0.5f, D);
  key = fmaf(D2 + c, inv, -R);
  lb = (D2 + c - kCullPad * (D2 + fabsf(me.w) + fabsf(lo.w))) * inv;
  return !(lb > R * (1.0f + 2.0f * kCullPad));
}

// Sign of the vertex of planes T (of `pid`) against site hpid's plane in FP64
// (see side64u): bit 0 outside, bit 1 still within its bound.
static __device__ __noinline__ unsigned walk_resolve64(const int* pid, uint32_t T, int hpid, float4 me,
                                                       const float* box, const float4* __restrict__ sites) {
  const Plane64u A = plane64u(pid[T & 255u], me, box, box + 3, sites);
  const Plane64u B = plane64u(pid[(T >> 8) & 255u], me, box, box + 3, sites);
  const Plane64u C = plane64u(pid[(T >> 16) & 255u], me, box, box + 3, sites);
  const Plane64u H = plane64u(hpid, me, box, box + 3, sites);
  bool a = false;
  const bool out = side64u(A, B, C, H, a);
  return (out ? 1u : 0u) | (a ? 2u : 0u);
}

// FP64 re-solve of a vertex, in place (see refine_vertex).
static __device__ __noinline__ void walk_refine(float4* v, int pa, int pb, int ph, float4 me, const float* box,
                                                const float4* __restrict__ sites) {
  float x, y, z, e;
  refine_vertex(pa, pb, ph, me, box, box + 3, sites, x, y, z, e);
  *v = make_float4(x, y, z, e);
}

}  // namespace vd
