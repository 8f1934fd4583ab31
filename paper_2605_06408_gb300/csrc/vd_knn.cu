// vd_knn.cu -- the K nearest sites of every site, by a query on the LBVH:
// the input of the KNN warm start of App. A.6, where each cell is first
// clipped by the planes of its K = 8 nearest sites, so that the directional
// bounds are tight from the first node test of the traversal on.
//
// Eight lanes per site, four sites per warp: a depth-first descent of the
// site's set's 8-wide tree, one child per lane, a leaf's (at most 16) sites
// two per lane; lane i of a group holds the group's i-th nearest site so far.
// The list starts with the site's eight neighbours in the sorted order, so
// that the first node tests already have a bound. A thread per site with the
// list in its registers (the earlier form) took a memory round trip for every
// site it read: 500 sites 77 -> 16 us, 10,000 148 -> 29 us, 1M 1.35 -> 1.15 ms
// (with log-normal weights 3.5 -> 2.2 ms), 20M 25 -> 22 ms.
//
// Any K sites give a valid warm start (clipping by any site's plane keeps the
// exact cell), so a stack that runs out of room only makes the list
// approximate, never wrong.
#include "vd_internal.cuh"

namespace vd {

namespace {

constexpr int kKnnStack = 48;
static_assert(kKnn == 8, "one list entry per lane of a group");

__device__ __forceinline__ float knn_min8(float v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(FULL, v, o));
  return v;
}

// Put (v, id) of lane `src` (one per group, where `in`) into the group's list.
__device__ __forceinline__ void knn_insert(float v, int id, int src, bool in, int gl, unsigned gsh, float& bd, int& bi) {
  v = __shfl_sync(FULL, v, src, 8);
  id = __shfl_sync(FULL, id, src, 8);
  const int pos = __popc((__ballot_sync(FULL, bd <= v) >> gsh) & 255u);  // sorted: the entries before it
  const float ud = __shfl_up_sync(FULL, bd, 1, 8);
  const int ui = __shfl_up_sync(FULL, bi, 1, 8);
  if (in && gl >= pos) {
    bd = gl == pos ? v : ud;
    bi = gl == pos ? id : ui;
  }
}

__global__ void __launch_bounds__(128) knn_kernel(const float4* __restrict__ sites, const float4* __restrict__ wide,
                                                  const SetInfo* __restrict__ sets, int nsets,
                                                  const uint64_t* __restrict__ keys, int set_shift,
                                                  const unsigned char* __restrict__ loser, int begin, int end,
                                                  int* __restrict__ knn) {
  __shared__ int sref[16][kKnnStack];
  __shared__ float sd[16][kKnnStack];
  const unsigned lane = lane_id();
  const int gl = (int)(lane & 7u), grp = (int)(threadIdx.x >> 3);
  const unsigned gsh = lane & 24u;
  const uint32_t ltg = (1u << gl) - 1u;
  const int want = begin + (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 3);
  const int si = min(want, end - 1);
  const float4 p = sites[si];
  // a loser of a duplicate position and a site that is not finite need no list
  // (and would find no bound to stop at)
  const bool own = want < end, live = own && loser[si] == 0 && finite_site(p);
  const SetInfo& SI = sets[nsets > 1 ? (int)(keys[si] >> set_shift) : 0];
  const int lo = SI.first, hi = SI.first + SI.count;
  const int w0 = max(lo, min(si - 4, hi - 9)), w1 = min(hi, w0 + 9);
  // the sorted neighbours, sorted by distance (an odd-even sort of 8)
  float bd = INFINITY;
  int bi = -1;
  {
    const int j = w0 + gl + (w0 + gl >= si ? 1 : 0);
    if (j < w1 && loser[j] == 0) {
      const float4 q = sites[j];
      const float dx = q.x - p.x, dy = q.y - p.y, dz = q.z - p.z;
      bd = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      bi = j;
    }
#pragma unroll
    for (int r = 0; r < 8; r++) {
      const bool low = ((gl ^ r) & 1) == 0;
      const int to = low ? gl + 1 : gl - 1;
      const float od = __shfl_sync(FULL, bd, to & 7, 8);
      const int oi = __shfl_sync(FULL, bi, to & 7, 8);
      if (to >= 0 && to < 8 && (low ? od < bd : od > bd)) {
        bd = od;
        bi = oi;
      }
    }
  }
  int top = 0;
  int cur = live ? SI.wroot : kNoChild;  // the node or leaf to visit next
  uint32_t pend = 0;                     // children of the node visited last that are leaves to read
  int cref = 0;
  float cd = 0.f;
  while (true) {
    const float bound = __shfl_sync(FULL, bd, 7, 8);
    if (cur == kNoChild && pend == 0 && top > 0) {
      top--;
      if (sd[grp][top] < bound) cur = sref[grp][top];
    }
    if (!__any_sync(FULL, cur != kNoChild || pend != 0 || top > 0)) break;
    const bool node = cur != kNoChild && !ref_is_leaf(cur);
    if (__any_sync(FULL, node)) {
      bool keep = false;
      if (node) {
        const float4* nd = wide + 16 * (size_t)cur + gl;
        const float4 l = __ldg(nd), h = __ldg(nd + 8);
        const float dx = fmaxf(fmaxf(l.x - p.x, p.x - h.x), 0.f), dy = fmaxf(fmaxf(l.y - p.y, p.y - h.y), 0.f),
                    dz = fmaxf(fmaxf(l.z - p.z, p.z - h.z), 0.f);
        cd = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        cref = __float_as_int(h.w);
        keep = cref != kNoChild && cd < bound;
      }
      const bool inner = keep && !ref_is_leaf(cref);
      const uint32_t im = (__ballot_sync(FULL, inner) >> gsh) & 255u;
      const uint32_t lm = (__ballot_sync(FULL, keep && !inner) >> gsh) & 255u;
      // the nearest inner child is next, the others go on the stack
      const float near = knn_min8(inner ? cd : INFINITY);
      const uint32_t nm = (__ballot_sync(FULL, inner && cd == near) >> gsh) & 255u;
      const int src = __ffs(nm) - 1;
      const int child = __shfl_sync(FULL, cref, src & 7, 8);
      if (node) {
        const uint32_t rest = im & ~(1u << (src & 31));
        if (inner && gl != src) {
          const int at = top + __popc(rest & ltg);
          if (at < kKnnStack) {
            sref[grp][at] = cref;
            sd[grp][at] = cd;
          }
        }
        top = min(kKnnStack, top + __popc(im ? rest : 0u));
        pend = lm;
        cur = kNoChild;
        if (im) {  // below the leaves: read them first, they tighten the bound
          if (lm == 0) {
            cur = child;
          } else if (top < kKnnStack) {
            if (gl == 0) {
              sref[grp][top] = child;
              sd[grp][top] = near;
            }
            top++;
          }
        }
      }
      __syncwarp();
      continue;
    }
    // a leaf: two sites per lane
    const bool root = cur != kNoChild;  // a set of one leaf
    const bool leaf = root || pend != 0;
    const int c = __ffs(pend) - 1;
    const int from = __shfl_sync(FULL, cref, c & 7, 8);
    const int ref = root ? cur : from;
    if (leaf && !root) pend &= pend - 1;
    cur = kNoChild;
    float d[2];
    int j[2];
#pragma unroll
    for (int r = 0; r < 2; r++) {
      const int k = gl + 8 * r;
      j[r] = leaf_first(ref) + k;
      const bool ok = leaf && k < leaf_count(ref) && (j[r] < w0 || j[r] >= w1);
      const int at = ok ? j[r] : si;
      const float4 q = sites[at];
      const unsigned char lost = loser[at];
      const float dx = q.x - p.x, dy = q.y - p.y, dz = q.z - p.z;
      d[r] = ok && lost == 0 ? fmaf(dx, dx, fmaf(dy, dy, dz * dz)) : INFINITY;
    }
    while (true) {
      const float b7 = __shfl_sync(FULL, bd, 7, 8);
      const float mine = fminf(d[0], d[1]);
      const float best = knn_min8(mine);
      const bool in = best < b7;
      if (!__any_sync(FULL, in)) break;
      const uint32_t bm = (__ballot_sync(FULL, mine == best) >> gsh) & 255u;
      const int src = __ffs(bm) - 1;
      const bool first = d[0] <= d[1];
      knn_insert(mine, first ? j[0] : j[1], src & 7, in, gl, gsh, bd, bi);
      if (in && gl == src) {
        if (first)
          d[0] = INFINITY;
        else
          d[1] = INFINITY;
      }
    }
  }
  if (own) knn[(size_t)si * kKnn + gl] = live ? bi : -1;
}

}  // namespace

cudaError_t launch_knn(const CellBuffers& c, int* knn, cudaStream_t s) {
  // the four cells that a warp of vd_quad.cu makes together, all of them
  const int begin = c.cell_begin & ~3, end = min((c.cell_end + 3) & ~3, c.n);
  const int m = end - begin;
  if (m <= 0) return cudaSuccess;
  knn_kernel<<<(int)((8ll * m + 127) / 128), 128, 0, s>>>(c.sites, c.wide, c.sets, c.nsets, c.keys, c.set_shift, c.loser,
                                                          begin, end, knn);
  return cudaGetLastError();
}

}  // namespace vd
