// vd_solo.cu -- the fused per-cell kernel, one cell per warp: the steps of
// vd_quad.cu with all 32 lanes on one cell. It makes the builds too small for
// four cells per warp (their time is the latency of one warp's work) and the
// cells that outgrow a group there.
//   T  pop up to four nodes of the 8-wide tree and test their 32 children,
//      read up to four leaves a step, 16 sites each, into the list of
//      candidates, until the list is long or the queue is empty;
//   F  one candidate per lane: its plane, and whether any vertex lies outside;
//   C  the nearest of those that cut, its plane broadcast, the vertices
//      classified, the removed ones listed;
//   H  the hole's edges and the new vertices (App. B).
// Measured against vd_cells.cu (as it was): 500 sites 98 -> 78 us, 10,000 430 ->
// 380 us; the cells that outgrow 48 vertices of 1M sites in clusters and the
// large-cell pass after it, 7.7 ms of that pass before -> 3.0 ms.
// Polytope, planes, queue and candidates are in shared memory (11 KB a warp);
// up to 192 vertices and 128 planes. Larger cells, and cells whose walk is long
// or outgrows the queue, go to the large-cell pass.
#include "vd_walk.cuh"

namespace vd {
namespace {

constexpr int kSV = 192;  // vertices (their slot takes a byte of otri)
constexpr int kSBrute = 128;  // vertices without a tree (larger cells are not made there)
constexpr int kSP = 128;  // planes (a byte of a triplet)
constexpr int kSQ = 96;   // queue entries (7 bits of the key)
constexpr int kSC = 96;   // candidates
constexpr int kST = 23;   // candidates at which the walk stops to clip (a step adds up to 64)
constexpr int kSF = 39;   // faces of a cell whose edges are looked up in a table at the end
constexpr int kSCone = 40;  // node visits (of up to four nodes) after which the cone test is made
// Node visits after which a cell goes to the large-cell pass. They take 4.6 us
// each, one warp at work on them long after the others (a cell at the hull of a
// tight cluster that sees the whole empty box); there up to eight warps share a
// cell's filters, and such sets have heavier cells in that pass anyway. Builds
// without a limit, with 2,000 and with 1,000: 300,000 sites in 0.1% of each side
// 194, 179 and 175 ms, in a ball of 5% 107.8, 109.1 and 106.6, one cluster of
// sigma 0.01 86.4, 78.8 and 77.4, five clusters 52.0, 48.9 and 46.2; but 20,000 on
// a shell 8.7, 8.7 and 18.3 (its only cell past 1,000 took 9.7 ms in that pass).
constexpr int kSWalk = 2000;
static_assert(kST + 1 + 64 <= kSC, "room for a step's leaves");

struct __align__(16) SoloCell {
  float4 vp[kSV];      // position, error bound; with pl the scratch of the FP64 integration
  float4 pl[kSP];      // n^, b^
  float4 cand[kSC];    // candidate sites; at the end the edge table
  float pe[kSP];       // offset error bound; the FP64 integration's face anchors
  int pid[kSP];        // sorted site index, or -1-f for box face f
  uint32_t vt[kSV];    // plane triplet
  uint32_t otri[kSV];  // triplets a clip removes (bits 24 up: their slots); at the end renumbered triplets
  int cid[kSC];
  uint32_t q[2 * kSQ];  // queue: ordered keys (17 bits, children to visit (8), free for the slot (7)), then nodes;
                        // at the end the neighbour list
  unsigned char fill[kSV];  // slots to fill
  uint32_t freep[kSP / 32];  // plane slots reclaimed once all have been used
  unsigned tally[4];  // of the warp's finished cells: FP64 signs, those still ambiguous, vertices re-solved
};
static_assert(kSF * kSF <= kSC * 16, "edge table over the candidates");
static_assert(sizeof(double) * 3 * kSV <= sizeof(float4) * (kSV + kSP), "FP64 scratch");

enum { S_BUILD = 0, S_EMPTY = 1, S_FULL = 2, S_FAR = 3, S_PLANES = 4, S_ROW = 5 };

// Volume and first moment about (cx, cy, cz) in FP64 (the scheme of
// volume_fp64). Overwrites vp, pl and pe.
struct SoloMoments {
  double v, x, y, z;
};
__device__ __noinline__ SoloMoments solo_volume64(SoloCell& S, int nv, float4 me, const float* box,
                                              const float4* __restrict__ sites, double cx, double cy, double cz) {
  const int lane = (int)lane_id();
  double* vd64 = reinterpret_cast<double*>(S.vp);
  int* anchor = reinterpret_cast<int*>(S.pe);
  for (int f = lane; f < kSP; f += 32) anchor[f] = 0x7fffffff;
  __syncwarp();
#pragma unroll 1
  for (int t = lane; t < nv; t += 32) {
    const uint32_t T = S.vt[t];
    double x, y, z;
    vertex64(T & 255u, (T >> 8) & 255u, (T >> 16) & 255u, S.pid, me, box, box + 3, sites, x, y, z);
    vd64[3 * t] = x - cx;
    vd64[3 * t + 1] = y - cy;
    vd64[3 * t + 2] = z - cz;
    atomicMin(&anchor[T & 255u], t);
    atomicMin(&anchor[(T >> 8) & 255u], t);
    atomicMin(&anchor[(T >> 16) & 255u], t);
  }
  __syncwarp();
  double V = 0.0, Mx = 0.0, My = 0.0, Mz = 0.0;
#pragma unroll 1
  for (int it = lane; it < 3 * nv; it += 32) {
    const int t = it / 3, rho = it - 3 * t;
    const uint32_t T = S.vt[t];
    const uint32_t xy = ((T | (T << 24)) >> (8 * rho)) & 0xffffu;
    const uint32_t fy = xy >> 8, q = fy | ((xy & 255u) << 8);
    int u = 0;
    while (u < nv && !tri_has_pair(S.vt[u], q)) u++;
    const int g = anchor[fy];
    if (u >= nv || g == t || g == u) continue;  // triangles through the anchor vanish
    const double* A = &vd64[3 * g];
    const double* B = &vd64[3 * t];
    const double* C = &vd64[3 * u];
    const double det = A[0] * (B[1] * C[2] - B[2] * C[1]) + A[1] * (B[2] * C[0] - B[0] * C[2]) +
                       A[2] * (B[0] * C[1] - B[1] * C[0]);
    V += det;
    Mx += det * (A[0] + B[0] + C[0]);
    My += det * (A[1] + B[1] + C[1]);
    Mz += det * (A[2] + B[2] + C[2]);
  }
  __syncwarp();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    V += __shfl_xor_sync(FULL, V, o);
    Mx += __shfl_xor_sync(FULL, Mx, o);
    My += __shfl_xor_sync(FULL, My, o);
    Mz += __shfl_xor_sync(FULL, Mz, o);
  }
  return SoloMoments{V / 6.0, Mx / 24.0, My / 24.0, Mz / 24.0};
}

// A plane slot that no vertex uses but the k about to be removed (otri), or
// -1. Called once every slot has been used.
__device__ __noinline__ int solo_reclaim(SoloCell& S, int nv, int k) {
  const int lane = (int)lane_id();
  uint32_t f = lane < kSP / 32 ? S.freep[lane] : 0u;
  uint32_t any = __ballot_sync(FULL, f != 0);
  if (!any) {
    uint32_t used[kSP / 32];
#pragma unroll
    for (int w = 0; w < kSP / 32; w++) used[w] = 0;
    for (int v = lane; v < nv; v += 32) {
      bool gone = false;
      for (int t = 0; t < k; t++) gone = gone || (int)(S.otri[t] >> 24) == v;
      if (gone) continue;
      const uint32_t T = S.vt[v];
#pragma unroll
      for (int c = 0; c < 3; c++) {
        const uint32_t p = (T >> (8 * c)) & 255u;
#pragma unroll
        for (int w = 0; w < kSP / 32; w++)
          if ((p >> 5) == (uint32_t)w) used[w] |= 1u << (p & 31u);
      }
    }
    __syncwarp();
#pragma unroll
    for (int w = 0; w < kSP / 32; w++) {
      const uint32_t u = __reduce_or_sync(FULL, used[w]);
      if (lane == w) f = ~u;
    }
    any = __ballot_sync(FULL, f != 0);
    if (!any) return -1;
  }
  const int w = __ffs(any) - 1;
  const uint32_t bits = __shfl_sync(FULL, f, w);
  if (lane == w) f &= f - 1;
  if (lane < kSP / 32) S.freep[lane] = f;
  __syncwarp();
  return 32 * w + __ffs(bits) - 1;
}

// After a clip that made m vertices for the k it removed, m < k: the slots
// left over are filled from the end of the array.
__device__ __noinline__ void solo_fill(SoloCell& S, int nv, int m, int k) {
  const int lane = (int)lane_id();
  const uint32_t lt = lanemask_lt();
  const int over = k - m, to = nv - over;
  for (int t = lane; t < over; t += 32) S.vt[S.otri[m + t] >> 24] = kEmptyTri;
  __syncwarp();
  int holes = 0, live = 0;
  for (int b0 = 0; b0 < over; b0 += 32) {
    const int t = b0 + lane;
    const int slot = t < over ? (int)(S.otri[m + t] >> 24) : kSV;
    const uint32_t hm = __ballot_sync(FULL, slot < to);
    if (slot < to) S.fill[holes + __popc(hm & lt)] = (unsigned char)slot;
    holes += __popc(hm);
  }
  __syncwarp();
  for (int b0 = 0; b0 < over; b0 += 32) {
    const int v = to + b0 + lane;
    const bool mv = b0 + lane < over && S.vt[v] != kEmptyTri;
    const uint32_t vm = __ballot_sync(FULL, mv);
    if (mv) {
      const int slot = S.fill[live + __popc(vm & lt)];
      S.vp[slot] = S.vp[v];
      S.vt[slot] = S.vt[v];
    }
    live += __popc(vm);
  }
  __syncwarp();
}

// May a site of the box [lo, hi] cut the cell of vertices vp, by the cone of
// directions toward the box (see node_cone) and the cell's support in the
// cone's axis, exact over the vertices?
__device__ __noinline__ bool solo_cone_test(const float4* vp, int nv, float4 lo, float4 hi, float4 me, float lb,
                                            float reach2) {
  Cone k;
  if (!node_cone(lo, hi, me, k)) return true;
  float h = -INFINITY, em = 0.f;
  for (int v = 0; v < nv; v++) {
    const float4 p = vp[v];
    h = fmaxf(h, fmaf(k.ux, p.x, fmaf(k.uy, p.y, k.uz * p.z)));
    em = fmaxf(em, p.w);
  }
  return !cone_culls(lb, h, em, sqrt_approx(reach2) * (1.0f + kCullPad), k);
}

// The cell's record for the adjoint (otri holds the renumbered triplets): the
// site's own (see write_tape in vd_cells.cu) or, when it is too large for
// that, one on the large-cell tape (see big_tape_write there).
__device__ __noinline__ void solo_tape(const SoloCell& S, const CellBuffers& P, int si, int nv, int nf, uint32_t a0,
                                       uint32_t a1, uint32_t a2, uint32_t a3) {
  const int lane = (int)lane_id();
  const uint32_t alive[4] = {a0, a1, a2, a3};
  char* head = P.tape + (size_t)si * kTapeStride;
  if (nv <= kTapeV && nf <= kTapeF) {
    float4* tv = reinterpret_cast<float4*>(head + kTapeVOff);
    for (int t = lane; t < nv; t += 32) {
      const float4 p = S.vp[t];
      tv[t] = make_float4(p.x, p.y, p.z, __uint_as_float(S.otri[t]));
    }
    int* tf = reinterpret_cast<int*>(head + kTapeFOff);
    int n = 0;
#pragma unroll
    for (int w = 0; w < 4; w++) {
      if ((alive[w] >> lane) & 1u) tf[n + __popc(alive[w] & ((1u << lane) - 1u))] = S.pid[32 * w + lane];
      n += __popc(alive[w]);
    }
    if (lane == 0) *reinterpret_cast<int4*>(head) = make_int4(nv, nf, 0, 0);
    return;
  }
  const long long bytes = big_tape_bytes(nv, nf);
  unsigned long long off = 0;
  if (P.btape && lane == 0) off = atomicAdd((unsigned long long*)&P.st->btape_used, (unsigned long long)bytes);
  off = __shfl_sync(FULL, off, 0);
  if (!P.btape || (long long)off + bytes > P.btape_cap) {
    if (lane == 0) *reinterpret_cast<int4*>(head) = make_int4(-1, nf, 0, 0);
    return;
  }
  char* rec = P.btape + off;
  float4* vp = reinterpret_cast<float4*>(rec + 16);
  uint64_t* vt = reinterpret_cast<uint64_t*>(rec + 16 + 16 * (size_t)nv);
  int* pid = reinterpret_cast<int*>(rec + 16 + 24 * (size_t)nv);
  for (int t = lane; t < nv; t += 32) {
    const uint32_t R = S.otri[t];
    vp[t] = S.vp[t];
    vt[t] = (uint64_t)(R & 255u) | ((uint64_t)((R >> 8) & 255u) << 16) | ((uint64_t)(R >> 16) << 32);
  }
  int n = 0;
#pragma unroll
  for (int w = 0; w < 4; w++) {
    if ((alive[w] >> lane) & 1u) pid[n + __popc(alive[w] & ((1u << lane) - 1u))] = S.pid[32 * w + lane];
    n += __popc(alive[w]);
  }
  if (lane == 0) {
    atomicAdd((unsigned long long*)&P.st->btape_records, 1ull);
    *reinterpret_cast<int4*>(rec) = make_int4(nv, nf, 0, 0);
    *reinterpret_cast<int4*>(head) = make_int4(-2, nf, (int)(unsigned)(off & 0xffffffffull), (int)(unsigned)(off >> 32));
  }
}

// Take the (up to four) best entries off the queue; each 8-lane group gets
// one of them and the children to visit, or -1.
__device__ __forceinline__ int solo_pop(SoloCell& S, int& qn, uint32_t& todo) {
  const int lane = (int)lane_id();
  const uint32_t lt = lanemask_lt();
  uint32_t k[3];
  int r[3];
  const int rounds = (qn + 31) >> 5;
#pragma unroll
  for (int t = 0; t < 3; t++) {
    k[t] = 0xffffffffu;
    r[t] = -1;
    if (t < rounds && lane + 32 * t < qn) {
      k[t] = S.q[lane + 32 * t] | (uint32_t)(lane + 32 * t);
      r[t] = S.q[kSQ + lane + 32 * t];
    }
  }
  // one at a time once the queue has grown: strictly best first keeps it short
  const int take = qn > 32 ? 1 : 4;
  int ref = -1;
#pragma unroll
  for (int g = 0; g < 4; g++) {
    if (g < take) {
      const uint32_t b = __reduce_min_sync(FULL, min(k[0], min(k[1], k[2])));
      if (b != 0xffffffffu) {
        if ((lane >> 3) == g) {
          ref = S.q[kSQ + (b & 127u)];
          todo = (b >> 7) & 255u;
        }
#pragma unroll
        for (int t = 0; t < 3; t++)
          if (k[t] == b) k[t] = 0xffffffffu;
      }
    }
  }
  __syncwarp();
  int n = 0;
#pragma unroll
  for (int t = 0; t < 3; t++) {
    if (t < rounds) {
      const bool live = k[t] != 0xffffffffu;
      const uint32_t m = __ballot_sync(FULL, live);
      if (live) {
        const int to = n + __popc(m & lt);
        S.q[to] = k[t] & ~127u;
        S.q[kSQ + to] = r[t];
      }
      n += __popc(m);
    }
  }
  qn = n;
  __syncwarp();
  return ref;
}

// BRUTE: no tree; every site of one set is read, 64 a step, after the nearest
// of every 32nd (one per lane) have clipped the cell (vd_cells_noalloc). A
// cell that does not fit is marked there and then.
template <bool BRUTE>
__global__ void __launch_bounds__(128, 4) solo_kernel(CellBuffers P) {
  extern __shared__ __align__(16) unsigned char solo_smem[];
  SoloCell& S = reinterpret_cast<SoloCell*>(solo_smem)[threadIdx.x >> 5];
  const int lane = (int)lane_id();
  const uint32_t lt = lanemask_lt();
  const float u = Num<float>::u;
  unsigned ctrefvol = 0, ctempty = 0, ctovf = 0;
  if (lane < 4) S.tally[lane] = 0;
  int* const work = P.from_mid ? &P.work[5] : &P.work[0];
  const int total = P.from_mid ? P.st->mid_count : P.cell_end - P.cell_begin;
  auto original = [&](int j) { return BRUTE ? j : P.perm[j]; };

  while (true) {
    int item = 0;
    if (lane == 0) item = atomicAdd(work, 1);
    item = __shfl_sync(FULL, item, 0);
    if (item >= total) break;
    const int si = P.from_mid ? P.mid_list[item] : P.cell_begin + item;
    const float4 me = P.sites[si];
    const int orig = original(si);
    const SetInfo& SI = P.sets[P.nsets > 1 ? (int)(P.keys[si] >> P.set_shift) : 0];
    const float* box = SI.lo;
    const bool weighted = SI.weighted != 0;
    int mode = P.loser[si] || !finite_site(me) ? S_EMPTY : S_BUILD;
    unsigned ct64 = 0, ctamb = 0, ctrefv = 0;  // this cell's, a lane's share

    // ---- the box: 6 planes, 8 corners (as init_cell)
    if (lane < 6) {
      const PlaneT<float> B = box_plane<float>(lane, me.x, me.y, me.z, box, box + 3);
      S.pl[lane] = make_float4(B.nx, B.ny, B.nz, B.b);
      S.pe[lane] = B.e;
      S.pid[lane] = -1 - lane;
    }
    if (lane == 0) {
      S.q[0] = 255u << 7;
      S.q[kSQ + 0] = SI.wroot;
    }
    if (lane < kSP / 32) S.freep[lane] = 0;
    __syncwarp();
    if (lane < 8) {
      const int sx = lane & 1, sy = (lane >> 1) & 1, sz = lane >> 2;
      const bool odd = (sx + sy + sz) & 1;
      const uint32_t b = odd ? 4 + sz : 2 + sy, d = odd ? 2 + sy : 4 + sz;
      const float px = S.pl[sx].w, py = S.pl[2 + sy].w, pz = S.pl[4 + sz].w;
      const float x = sx ? -px : px, y = sy ? -py : py, z = sz ? -pz : pz;
      const float x1 = fabsf(x) + fabsf(y) + fabsf(z);
      const float ep = 1.75f * (S.pe[sx] + S.pe[2 + sy] + S.pe[4 + sz]) + (5.25f * 8.0f * u + 9.0f * u) * x1 +
                       6.0f * u * x1 + u * x1;
      S.vp[lane] = make_float4(x, y, z, x1 < 1e30f ? 1.1f * ep + 11.0f * u * x1 : INFINITY);
      S.vt[lane] = (uint32_t)sx | (b << 8) | (d << 16);
    }
    int nv = 8, np = 6, qn = 1, cn = 0;

    // ---- first sites: the KNN list (App. A.6)
    int kid = -1;
    if (BRUTE) {
      float best = INFINITY;
      for (int j = lane; j < P.n; j += 32) {
        const float4 q = P.sites[j];
        const float dx = q.x - me.x, dy = q.y - me.y, dz = q.z - me.z;
        const float d = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) - q.w;
        if (d < best && j != si) {
          best = d;
          kid = j;
        }
      }
    } else if (lane < kKnn) {
      kid = P.knn[(size_t)si * kKnn + lane];
    }
    {
      const uint32_t m = __ballot_sync(FULL, kid >= 0);
      if (kid >= 0) {
        const int at = __popc(m & lt);
        S.cand[at] = P.sites[kid];
        S.cid[at] = kid;
      }
      cn = __popc(m);
    }
    __syncwarp();
    int cur = -1;       // the node to visit next, if it is not the queue's best
    uint32_t pend = 0;  // lanes whose child of the nodes visited last is a leaf still to be read
    int cref = 0;
    bool first = true, finished = false, dirty = true;
    int steps = 0;  // node visits of the walk (BRUTE: sites read)
    WalkBounds B;

#pragma unroll 1
    while (mode == S_BUILD) {
      // ---- A: bounds of the polytope
      if (dirty) {
        float mn0 = INFINITY, mn1 = INFINITY, mn2 = INFINITY, mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY;
        float em = 0.f;
#pragma unroll 1
        for (int v = lane; v < nv; v += 32) {
          const float4 p = S.vp[v];
          mn0 = fminf(mn0, p.x);
          mn1 = fminf(mn1, p.y);
          mn2 = fminf(mn2, p.z);
          mx0 = fmaxf(mx0, p.x);
          mx1 = fmaxf(mx1, p.y);
          mx2 = fmaxf(mx2, p.z);
          em = fmaxf(em, p.w);
        }
        __syncwarp();
        em = warp_maxf(em);
        B.lo[0] = warp_minf(mn0) - em;
        B.lo[1] = warp_minf(mn1) - em;
        B.lo[2] = warp_minf(mn2) - em;
        B.hi[0] = warp_maxf(mx0) + em;
        B.hi[1] = warp_maxf(mx1) + em;
        B.hi[2] = warp_maxf(mx2) + em;
#pragma unroll
        for (int k = 0; k < 3; k++) {
          B.lo2[k] = B.lo[k] * B.lo[k];
          B.hi2[k] = B.hi[k] * B.hi[k];
          B.c[k] = 0.5f * (B.lo[k] + B.hi[k]);
        }
        float r2 = 0.f;
#pragma unroll 1
        for (int v = lane; v < nv; v += 32) {
          const float4 p = S.vp[v];
          const float dx = p.x - B.c[0], dy = p.y - B.c[1], dz = p.z - B.c[2];
          r2 = fmaxf(r2, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        }
        __syncwarp();
        B.rad = (sqrt_approx(warp_maxf(r2)) + em) * (1.0f + kCullPad);
        const float reach = sqrt_approx(B.c[0] * B.c[0] + B.c[1] * B.c[1] + B.c[2] * B.c[2]) + B.rad;
        B.reach2 = reach * reach;
        B.ext = 4.0f * (reach + fabsf(B.c[0]) + fabsf(B.c[1]) + fabsf(B.c[2]) + B.rad);
        dirty = false;
      }

      // ---- T: walk until the list is long or nothing is left
#pragma unroll 1
      while (!first && cn <= kST) {
        float4 q[2];
        int j[2];
        bool act[2], keep[2];
        if constexpr (BRUTE) {
          if (steps >= P.n) {
            finished = true;
            break;
          }
#pragma unroll
          for (int r = 0; r < 2; r++) {
            j[r] = steps + 32 * r + lane;
            act[r] = (j[r] < P.n) & (j[r] != si);
            q[r] = P.sites[act[r] ? j[r] : si];
          }
          steps += 64;
        } else {
          if (pend == 0) {
            if (qn == 0 && cur < 0) {
              finished = true;
              break;
            }
            if (++steps > kSWalk) {
              mode = S_FAR;
              break;
            }
            uint32_t todo = 255u;
            int ref = lane < 8 ? cur : -1;
            if (cur < 0) ref = solo_pop(S, qn, todo);
            cur = -1;
            bool keep = false;
            float key = 0.f;
            if (ref >= 0) {
              const float4* nd = P.wide + 16 * (size_t)ref + (lane & 7);
              const float4 lo = __ldg(nd), hi = __ldg(nd + 8);
              cref = __float_as_int(hi.w);
              float lb;
              keep = walk_node_test(lo, hi, me, B, weighted, key, lb) && cref != kNoChild && ((todo >> (lane & 7)) & 1u);
              // a long walk: test the cone of directions toward the box too (see
              // node_cone), against the cell's exact support in the cone's axis
              if (steps > kSCone && keep) keep = solo_cone_test(S.vp, nv, lo, hi, me, lb, B.reach2);
            } else {  // none, or a set of one leaf
              cref = SI.wroot;
              keep = lane == 0 && ref_is_leaf(cref);
            }
            pend = __ballot_sync(FULL, keep && ref_is_leaf(cref));
            const bool inner = keep && !ref_is_leaf(cref);
            const uint32_t im = __ballot_sync(FULL, inner);
            if (im && qn + __popc(im) > kSQ - 24) {
              // little room (bounds still loose in several directions; one node
              // was visited): go on with the best child, and queue the node
              // itself with the others, to be tested again under the bounds of
              // that time
              const uint32_t kk = inner ? f2o(key) & ~0x7fffu : 0xffffffffu;
              const uint32_t b1 = __reduce_min_sync(FULL, inner ? (kk | (uint32_t)lane) : 0xffffffffu);
              const int src = (int)(b1 & 31u);
              const uint32_t rest = im & ~(1u << src);
              cur = __shfl_sync(FULL, cref, src);
              if (rest) {
                if (qn >= kSQ || im > 255u) {
                  mode = S_FAR;
                  break;
                }
                const uint32_t b2 = __reduce_min_sync(FULL, lane != src ? kk : 0xffffffffu);
                if (lane == 0) {
                  S.q[qn] = (b2 & ~0x7fffu) | (rest << 7);
                  S.q[kSQ + qn] = ref;
                }
                qn++;
              }
              __syncwarp();
              continue;
            }
            if (inner) {
              const int to = qn + __popc(im & lt);
              S.q[to] = (f2o(key) & ~0x7fffu) | (255u << 7);
              S.q[kSQ + to] = cref;
            }
            qn += __popc(im);
            __syncwarp();
            continue;
          }
          // read up to four leaves, two at a time
#pragma unroll
          for (int r = 0; r < 2; r++) {
            const int c0 = __ffs(pend) - 1;
            const uint32_t p1 = pend & (pend - 1);
            const int c1 = __ffs(p1) - 1;
            pend = p1 & (p1 - 1);
            const int c = lane < 16 ? c0 : c1;
            const int ref = __shfl_sync(FULL, cref, c & 31);
            j[r] = leaf_first(ref) + (lane & 15);
            act[r] = (c >= 0) & ((lane & 15) < leaf_count(ref)) & (j[r] != si);
            q[r] = P.sites[act[r] ? j[r] : si];
          }
        }
        bool dup = false;
#pragma unroll
        for (int r = 0; r < 2; r++) {
          const float nx = q[r].x - me.x, ny = q[r].y - me.y, nz = q[r].z - me.z;
          const float nn = fmaf(nx, nx, fmaf(ny, ny, nz * nz));
          keep[r] = act[r] & walk_site_test(nx, ny, nz, nn, me.w, q[r].w, B);
          dup = dup | (act[r] & (nn == 0.f));
        }
        if (__any_sync(FULL, dup)) {
          // duplicate positions (of another weight stratum: gather_sites sees
          // the others): the larger weight, then the lower index, wins
          bool lose = false;
#pragma unroll
          for (int r = 0; r < 2; r++)
            if (act[r] && q[r].x == me.x && q[r].y == me.y && q[r].z == me.z) {
              keep[r] = false;
              lose = lose || q[r].w > me.w || (q[r].w == me.w && original(j[r]) < orig);
            }
          if (__any_sync(FULL, lose)) {
            mode = S_EMPTY;
            break;
          }
        }
#pragma unroll
        for (int r = 0; r < 2; r++) {
          const uint32_t km = __ballot_sync(FULL, keep[r]);
          if (keep[r]) {
            const int at = cn + __popc(km & lt);
            S.cand[at] = q[r];
            S.cid[at] = j[r];
          }
          cn += __popc(km);
        }
      }
      if (mode != S_BUILD) break;
      __syncwarp();

#pragma unroll 1
      for (int base = 0; base < cn && mode == S_BUILD; base += 32) {
        // ---- F: the plane of each candidate, and whether it cuts the polytope
        PlaneT<float> H;
        H.nx = H.ny = H.nz = H.b = H.e = 0.f;
        int id = -1;
        bool left = base + lane < cn;
        if (left) {
          const float4 q = S.cand[base + lane];
          id = S.cid[base + lane];
          const float nx = q.x - me.x, ny = q.y - me.y, nz = q.z - me.z;
          if (P.loser[id]) left = false;
          if (first && nx == 0.f && ny == 0.f && nz == 0.f) {  // a duplicate position among the first sites
            if (left && (q.w > me.w || (q.w == me.w && original(id) < orig))) mode = S_EMPTY;
            left = false;
          }
          if (left) H = site_plane<float>(me.x, me.y, me.z, me.w, q.x, q.y, q.z, q.w);
        }
        if (__any_sync(FULL, mode == S_EMPTY)) {
          mode = S_EMPTY;
          break;
        }
        if (BRUTE && !first) left = left & (id != __shfl_sync(FULL, kid, id & 31));
        if (!BRUTE && !first) {
#pragma unroll
          for (int k = 0; k < kKnn; k++) left = left & (id != __shfl_sync(FULL, kid, k));
        }
        {
          // the sign test's value plus both error bounds (a little more of each
          // than the classification takes), as one chain per vertex
          const float nb = fmaf(1.25f, H.e, -H.b);
          float top = -INFINITY;
#pragma unroll 4
          for (int v = 0; v < nv; v++) {
            const float4 p = S.vp[v];
            top = fmaxf(top, fmaf(H.nx, p.x, fmaf(H.ny, p.y, fmaf(H.nz, p.z, fmaf(1.0001f, p.w, nb)))));
          }
          left = left & (top > 0.f);
        }
#pragma unroll 1
        while (__any_sync(FULL, left)) {
          // ---- C: the nearest one; classify the vertices, list the removed ones
          const uint32_t kk = left ? f2o(H.b) : 0xffffffffu;
          const uint32_t mn = __reduce_min_sync(FULL, kk);
          const int src = __ffs(__ballot_sync(FULL, left && kk == mn)) - 1;
          if (lane == src) left = false;
          PlaneT<float> G;
          G.nx = __shfl_sync(FULL, H.nx, src);
          G.ny = __shfl_sync(FULL, H.ny, src);
          G.nz = __shfl_sync(FULL, H.nz, src);
          G.b = __shfl_sync(FULL, H.b, src);
          G.e = __shfl_sync(FULL, H.e, src);
          const int hj = __shfl_sync(FULL, id, src);
          int k = 0;
#pragma unroll 1
          for (int b0 = 0; b0 < nv; b0 += 32) {
            const int v = b0 + lane;
            bool out = false, amb = false;
            if (v < nv) {
              const float4 p = S.vp[v];
              const float s = side<float>(G, p.x, p.y, p.z);
              out = s > 0.f;
              amb = ambiguous<float>(s, p.w, G.e);
            }
            if (__any_sync(FULL, amb)) {
              if (amb) {
                ct64++;
                const unsigned r = walk_resolve64(S.pid, S.vt[v], hj, me, box, P.sites);
                out = r & 1u;
                ctamb += r >> 1;
              }
              __syncwarp();
            }
            const uint32_t om = __ballot_sync(FULL, out);
            if (out) S.otri[k + __popc(om & lt)] = S.vt[v] | ((uint32_t)v << 24);
            k += __popc(om);
          }
          __syncwarp();  // the list: read by other lanes in solo_reclaim already
          if (k == 0) continue;
          if (k == nv) {
            mode = S_EMPTY;
            break;
          }
          // ---- H: a plane slot (slots no kept vertex uses are reclaimed when all are taken)
          int h = np;
          if (np < kSP) {
            np++;
          } else {
            h = solo_reclaim(S, nv, k);
            if (h < 0) {
              mode = S_PLANES;
              break;
            }
          }
          if (lane == 0) {
            S.pl[h] = make_float4(G.nx, G.ny, G.nz, G.b);
            S.pe[h] = G.e;
            S.pid[h] = hj;
          }
          __syncwarp();
          // the hole's edges: every directed pair (a, b) of a removed vertex whose
          // reverse is in no other removed vertex -> vertex (a, b, h). New vertex
          // t takes the slot of removed vertex t, then slots at the end
          int m = 0;
#pragma unroll 1
          for (int b0 = 0; b0 < k; b0 += 32) {
            const int t = b0 + lane;
            const bool own = t < k;
            const uint32_t T = own ? S.otri[t] : 0u;
            const uint32_t a = T & 255u, b = (T >> 8) & 255u, c = (T >> 16) & 255u;
            const uint32_t r0 = b | (a << 8), r1 = c | (b << 8), r2 = a | (c << 8);
            bool e0 = own, e1 = own, e2 = own;
#pragma unroll 2
            for (int v = 0; v < k; v++) {
              const uint32_t U = S.otri[v];
              const uint32_t p0 = U & 0xffffu, p1 = (U >> 8) & 0xffffu, p2 = ((U >> 16) & 255u) | ((U & 255u) << 8);
              e0 = e0 & (p0 != r0) & (p1 != r0) & (p2 != r0);
              e1 = e1 & (p0 != r1) & (p1 != r1) & (p2 != r1);
              e2 = e2 & (p0 != r2) & (p1 != r2) & (p2 != r2);
            }
            const uint32_t m0 = __ballot_sync(FULL, e0), m1 = __ballot_sync(FULL, e1), m2 = __ballot_sync(FULL, e2);
            int at = m + __popc(m0 & lt) + __popc(m1 & lt) + __popc(m2 & lt);
#pragma unroll
            for (int e = 0; e < 3; e++) {
              const bool is = e == 0 ? e0 : (e == 1 ? e1 : e2);
              const uint32_t ab = e == 0 ? (a | (b << 8)) : (e == 1 ? (b | (c << 8)) : (c | (a << 8)));
              if (is) {
                const int slot = at < k ? (int)(S.otri[at] >> 24) : nv + (at - k);
                if (slot < (BRUTE ? kSBrute : kSV)) S.vt[slot] = ab | ((uint32_t)h << 16);
                at++;
              }
            }
            m += __popc(m0) + __popc(m1) + __popc(m2);
          }
          if (nv - k + m > (BRUTE ? kSBrute : kSV)) {
            mode = S_FULL;
            break;
          }
          __syncwarp();
#pragma unroll 1
          for (int t = lane; t < m; t += 32) {
            const int slot = t < k ? (int)(S.otri[t] >> 24) : nv + (t - k);
            const uint32_t T = S.vt[slot];
            const int a = (int)(T & 255u), b = (int)((T >> 8) & 255u);
            const float4 pa = S.pl[a], pb = S.pl[b];
            PlaneT<float> A, C;
            A.nx = pa.x, A.ny = pa.y, A.nz = pa.z, A.b = pa.w, A.e = S.pe[a];
            C.nx = pb.x, C.ny = pb.y, C.nz = pb.z, C.b = pb.w, C.e = S.pe[b];
            float x, y, z, ev;
            vertex3<float>(A, C, G, x, y, z, ev);
            S.vp[slot] = make_float4(x, y, z, ev);
            if (!(ev <= kRefineRel * (fabsf(x) + fabsf(y) + fabsf(z)))) {
              walk_refine(&S.vp[slot], S.pid[a], S.pid[b], hj, me, box, P.sites);
              ctrefv++;
            }
          }
          __syncwarp();
          if (m < k) solo_fill(S, nv, m, k);
          nv += m - k;
          dirty = true;
        }
      }
      __syncwarp();  // the candidates have been read: the walk puts others in their places
      cn = 0;
      first = false;
      if (finished) break;
    }
    __syncwarp();

    // ---- outputs
    if (mode == S_BUILD) {
      if (dirty) {  // L below: the vertices' box about the site
        float mx = 0.f, my = 0.f, mz = 0.f;
        for (int v = lane; v < nv; v += 32) {
          const float4 p = S.vp[v];
          mx = fmaxf(mx, fabsf(p.x) + p.w);
          my = fmaxf(my, fabsf(p.y) + p.w);
          mz = fmaxf(mz, fabsf(p.z) + p.w);
        }
        __syncwarp();
        mx = warp_maxf(mx), my = warp_maxf(my), mz = warp_maxf(mz);
        B.hi2[0] = B.lo2[0] = mx * mx;
        B.hi2[1] = B.lo2[1] = my * my;
        B.hi2[2] = B.lo2[2] = mz * mz;
      }
      float sx = 0.f, sy = 0.f, sz = 0.f, emax = 0.f;
      uint32_t alive[kSP / 32];
#pragma unroll
      for (int w = 0; w < kSP / 32; w++) alive[w] = 0;
#pragma unroll 1
      for (int v = lane; v < nv; v += 32) {
        const float4 p = S.vp[v];
        const uint32_t T = S.vt[v];
        sx += p.x;
        sy += p.y;
        sz += p.z;
        emax = fmaxf(emax, p.w);
#pragma unroll
        for (int c = 0; c < 3; c++) {
          const uint32_t f = (T >> (8 * c)) & 255u;
#pragma unroll
          for (int w = 0; w < kSP / 32; w++)
            if ((f >> 5) == (uint32_t)w) alive[w] |= 1u << (f & 31u);
        }
      }
      __syncwarp();
      int pre[kSP / 32], nf = 0, nb = 0;
#pragma unroll
      for (int w = 0; w < kSP / 32; w++) {
        alive[w] = __reduce_or_sync(FULL, alive[w]);
        pre[w] = nf;
        nf += __popc(alive[w]);
      }
      sx = warp_sumf(sx);
      sy = warp_sumf(sy);
      sz = warp_sumf(sz);
      emax = warp_maxf(emax);
      // neighbours: site planes that carry a face, ascending
      uint32_t* list = S.q;
#pragma unroll
      for (int w = 0; w < kSP / 32; w++) {
        const int f = 32 * w + lane;
        const bool isn = ((alive[w] >> lane) & 1u) && S.pid[f] >= 0;
        const uint32_t mk = __ballot_sync(FULL, isn);
        if (isn) list[nb + __popc(mk & lt)] = (uint32_t)(original(S.pid[f]) - SI.first);
        nb += __popc(mk);
      }
      __syncwarp();
      // a list longer than a row goes to the pool
      int* row = P.scratch + (size_t)orig * P.stride;
      if (BRUTE && nb > P.stride) mode = S_ROW;
      if (!BRUTE && nb > P.stride) {
        unsigned long long off = 0;
        if (lane == 0) off = atomicAdd((unsigned long long*)&P.st->pool_used, (unsigned long long)nb);
        off = __shfl_sync(FULL, off, 0);
        if ((long long)off + nb > P.pool_cap) {
          mode = S_ROW;
        } else {
          row = P.pool + off;
          if (lane == 0) P.ovf_slot[orig] = (int)off;
        }
      }
      if (mode == S_BUILD) {
#pragma unroll 1
        for (int t = lane; t < nb; t += 32) {
          const int v = (int)list[t];
          int rank = 0;
#pragma unroll 4
          for (int w = 0; w < nb; w++) rank += (int)list[w] < v;
          row[rank] = v;
        }
        // triplets in the order of the planes that carry a face (otri), and the
        // vertex each directed plane pair belongs to: an edge's other end
        unsigned char* succ = reinterpret_cast<unsigned char*>(S.cand);
        const bool direct = nf <= kSF;
        auto rank_of = [&](uint32_t f) -> uint32_t {
          uint32_t r = 0;
#pragma unroll
          for (int w = 0; w < kSP / 32; w++)
            if ((f >> 5) == (uint32_t)w) r = (uint32_t)pre[w] + __popc(alive[w] & ((1u << (f & 31u)) - 1u));
          return r;
        };
#pragma unroll 1
        for (int v = lane; v < nv; v += 32) {
          const uint32_t T = S.vt[v];
          const uint32_t a = rank_of(T & 255u), b = rank_of((T >> 8) & 255u), c = rank_of((T >> 16) & 255u);
          S.otri[v] = a | (b << 8) | (c << 16);
          if (direct) {
            succ[a * kSF + b] = (unsigned char)v;
            succ[b * kSF + c] = (unsigned char)v;
            succ[c * kSF + a] = (unsigned char)v;
          }
        }
        __syncwarp();
        if (!BRUTE && P.tape) solo_tape(S, P, si, nv, nf, alive[0], alive[1], alive[2], alive[3]);
        __syncwarp();
        // volume and first moment: tetrahedra (c, g_f, v, w) as in cell_outputs
        const float inv = 1.0f / (float)nv;
        const float cx = sx * inv, cy = sy * inv, cz = sz * inv;
        float V = 0.f, Mx = 0.f, My = 0.f, Mz = 0.f, Sabs = 0.f;
#pragma unroll 1
        for (int it = lane; it < 3 * nv; it += 32) {
          const int t = it / 3, rho = it - 3 * t;
          const uint32_t T = S.vt[t], R = S.otri[t];
          const uint32_t fy = ((T | (T << 24)) >> (8 * rho + 8)) & 255u;
          const uint32_t xy = ((R | (R << 24)) >> (8 * rho)) & 0xffffu, x = xy & 255u, y = xy >> 8;
          int w = 0;
          if (direct)
            w = succ[y * kSF + x];
          else
            while (w < nv && !tri_has_pair(S.otri[w], y | (x << 8))) w++;
          if (w >= nv) continue;  // cannot happen for a closed polytope
          const float4 pf = S.pl[fy];
          const float hgt = fmaf(pf.x, cx, fmaf(pf.y, cy, fmaf(pf.z, cz, -pf.w)));
          const float gx = -hgt * pf.x, gy = -hgt * pf.y, gz = -hgt * pf.z;  // g_f - c
          const float4 a = S.vp[t], b = S.vp[w];
          const float ax = a.x - cx, ay = a.y - cy, az = a.z - cz;
          const float bx = b.x - cx, by = b.y - cy, bz = b.z - cz;
          const float det = gx * (ay * bz - az * by) + gy * (az * bx - ax * bz) + gz * (ax * by - ay * bx);
          V += det;
          Mx += det * (gx + ax + bx);
          My += det * (gy + ay + by);
          Mz += det * (gz + az + bz);
          const float e1x = ax - gx, e1y = ay - gy, e1z = az - gz, e2x = bx - gx, e2y = by - gy, e2z = bz - gz;
          const float crx = e1y * e2z - e1z * e2y, cry = e1z * e2x - e1x * e2z, crz = e1x * e2y - e1y * e2x;
          Sabs += sqrtf(crx * crx + cry * cry + crz * crz);
        }
        __syncwarp();
        V = warp_sumf(V) * (1.0f / 6.0f);
        Mx = warp_sumf(Mx) * (1.0f / 24.0f);
        My = warp_sumf(My) * (1.0f / 24.0f);
        Mz = warp_sumf(Mz) * (1.0f / 24.0f);
        Sabs = warp_sumf(Sabs) * 0.5f;
        float L = 0.f;
#pragma unroll
        for (int c = 0; c < 3; c++) L += fmaxf(B.lo2[c], B.hi2[c]);
        L = sqrtf(L);
        double ox = cx, oy = cy, oz = cz, Vd = V;
        if (volume_needs_fp64(V, L, Sabs, emax)) {
          const SoloMoments r = solo_volume64(S, nv, me, box, P.sites, (double)cx, (double)cy, (double)cz);
          Vd = r.v;
          if (Vd > 0.0) {
            const double iv = 1.0 / Vd;
            ox += r.x * iv;
            oy += r.y * iv;
            oz += r.z * iv;
          }
          if (lane == 0) ctrefvol++;
        } else if (V > 0.0f) {
          ox += Mx / V;
          oy += My / V;
          oz += Mz / V;
        }
        if (lane == 0) {
          P.counts[orig] = nb;
          P.vol[orig] = (float)Vd;
          P.cen[3 * (size_t)orig] = (float)((double)me.x + ox);
          P.cen[3 * (size_t)orig + 1] = (float)((double)me.y + oy);
          P.cen[3 * (size_t)orig + 2] = (float)((double)me.z + oz);
        }
      }
    }
    if (mode == S_EMPTY && lane == 0) {
      ctempty++;
      P.counts[orig] = 0;
      P.vol[orig] = 0.0f;
      P.cen[3 * (size_t)orig] = me.x;
      P.cen[3 * (size_t)orig + 1] = me.y;
      P.cen[3 * (size_t)orig + 2] = me.z;
    }
    if (BRUTE && mode > S_EMPTY && lane == 0) {
      const float nan = __int_as_float(0x7fc00000);
      P.counts[orig] = -1;
      P.vol[orig] = nan;
      P.cen[3 * (size_t)orig] = nan;
      P.cen[3 * (size_t)orig + 1] = nan;
      P.cen[3 * (size_t)orig + 2] = nan;
      set_error(P.st, VD_ERR_CELL_OVERFLOW);
    }
    if (!BRUTE && mode > S_EMPTY && lane == 0) {  // to the large-cell pass
      const int reason = mode == S_FULL     ? OVF_VERTICES
                         : mode == S_FAR    ? OVF_QUEUE
                         : mode == S_PLANES ? OVF_PLANES
                                            : OVF_NEIGHBORS;
      ctovf++;
      atomicAdd((unsigned long long*)&P.st->ovf_reason[reason], 1ull);
      P.ovf_list[atomicAdd(&P.st->ovf_count, 1)] = si;
      if (P.tape) *reinterpret_cast<int4*>(P.tape + (size_t)si * kTapeStride) = make_int4(-1, 0, 0, 0);
    }
    // the events of cells that this kernel finishes: those of one passed on are
    // counted by the large-cell pass
    if (mode <= S_EMPTY) {
      if (!BRUTE && __any_sync(FULL, ctamb != 0) && lane == 0) record_ambiguous(P.st, P.amb_list, P.amb_cap, orig);
      if (ctrefv) atomicAdd(&S.tally[2], ctrefv);
      if (ct64) {
        atomicAdd(&S.tally[0], ct64);
        atomicAdd(&S.tally[1], ctamb);
      }
    }
    __syncwarp();
  }
  if (lane == 0) {
    const unsigned ct64 = S.tally[0], ctamb = S.tally[1], ctrefv = S.tally[2];
    if (ct64) atomicAdd((unsigned long long*)&P.st->fp64_fallbacks, (unsigned long long)ct64);
    if (ctamb) atomicAdd((unsigned long long*)&P.st->fp64_ambiguous, (unsigned long long)ctamb);
    if (ctrefv) atomicAdd((unsigned long long*)&P.st->refined_vertices, (unsigned long long)ctrefv);
    if (ctrefvol) atomicAdd((unsigned long long*)&P.st->refined_volumes, (unsigned long long)ctrefvol);
    if (ctempty) atomicAdd((unsigned long long*)&P.st->empty_cells, (unsigned long long)ctempty);
    if (ctovf) atomicAdd((unsigned long long*)&P.st->overflow_cells, (unsigned long long)ctovf);
  }
}

}  // namespace

cudaError_t launch_solo(const CellBuffers& c, int num_sms, cudaStream_t s) {
  const int wpb = c.cfg.warps_per_block > 4 ? 4 : c.cfg.warps_per_block;
  const size_t smem = sizeof(SoloCell) * (size_t)wpb;
  cudaError_t err = cudaFuncSetAttribute(solo_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  int per_sm = c.cfg.blocks_per_sm;
  if (per_sm <= 0) {
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, solo_kernel<false>, 32 * wpb, smem);
    if (err != cudaSuccess) return err;
    if (per_sm <= 0) per_sm = 1;
  }
  solo_kernel<false><<<num_sms * per_sm, 32 * wpb, smem, s>>>(c);
  return cudaGetLastError();
}

// Through cudaLaunchKernel: its return value is this launch's own status.
cudaError_t launch_solo_brute(const CellBuffers& c, int num_sms, cudaStream_t s) {
  constexpr int wpb = 4;
  constexpr size_t smem = sizeof(SoloCell) * wpb;
  static_assert(smem <= 48 * 1024, "no attribute to set");
  int blocks = (c.n + wpb - 1) / wpb;
  if (num_sms > 0 && blocks > 4 * num_sms) blocks = 4 * num_sms;
  CellBuffers arg = c;
  void* args[] = {(void*)&arg};
  return cudaLaunchKernel((const void*)solo_kernel<true>, dim3(blocks), dim3(32 * wpb), args, smem, s);
}

}  // namespace vd
