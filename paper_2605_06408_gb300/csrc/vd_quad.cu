// vd_quad.cu -- the fused per-cell kernel, four cells per warp: best-first
// traversal (Alg. 1), culling (Sec. 4.2), clipping (Sec. 4.1, App. B) and the
// cell's outputs, with 8 lanes per cell.
//
// What bounds this path is the number of warp instructions and the latency
// of one cell's chain of dependent steps, not memory: a cell has about 27
// vertices, 16 faces and 120 node tests. On 32 lanes per cell (vd_cells.cu)
// most lanes idle in every step: 25 vertices on 64 slots, two node children,
// five new vertices a clip, a few survivors a leaf. Here the four 8-lane
// groups of a warp each hold one of four consecutive cells of the sorted
// order, which need nearly the same part of the tree, and share one walk of
// an 8-wide tree:
//   A  refresh the bounds of the polytopes (vertex box, sphere);
//   T  pop the best node of the warp's queue and test its 8 children (one
//      per lane) for the four cells at once; read the leaves that some cell
//      needs, one site per lane, into each cell's list of candidate planes,
//      until a list is nearly full or the queue is empty;
//   F  drop the candidates that leave every vertex of the cell inside (one
//      candidate per lane);
//   C  take each cell's nearest candidate and classify its vertices, until
//      one cuts;
//   H  clip (all groups that found one).
// Measured against one warp per cell (vd_cells.cu, as it was): 300,000
// uniform sites 9.9 -> 5.2 ms, 1M in clusters 40.5 -> 24.4 ms, 2M on surfaces
// 92 -> 58 ms; warp instructions a cell 22,000 -> 12,700 (uniform) and
// 29,000 -> 18,900 (surfaces).
// Every collective runs on the whole warp and every loop ends on a warp vote
// or a warp-uniform count (a group without work is masked).
//
// Cells that outgrow the group's capacity (48 vertices, 48 planes) and cells
// whose walk is long (a cell that faces empty space reaches far; that kernel
// also tests nodes by their cone of directions) are listed for the
// one-cell-per-warp kernel of vd_solo.cu.
#include "vd_walk.cuh"

namespace vd {
namespace {

constexpr int kQV = 48;  // vertices per cell
constexpr int kQP = 48;  // planes per cell
constexpr int kQQ = 96;  // queue entries (inner nodes) per warp; the slot shares a word with the key
constexpr int kQC = 32;   // candidate planes of a cell collected before it is clipped by them
constexpr int kQT = 16;   // candidates at which the walk stops to clip (a leaf adds up to 16)
constexpr int kQS = 8;    // cutting candidates at which the cells are clipped before the walk goes on
static_assert(kQT + 16 <= kQC, "room for a leaf");
constexpr int kQF = 27;    // faces of a cell whose edges are looked up in a table at the end
constexpr int kQN = 400;   // nodes that a quad visits before its cells go elsewhere (45 on uniform sites, 80 on clusters
                           // and surfaces)
constexpr int kQLeafRoot = (1 << 26) - 1;  // queue reference of a set of one leaf
constexpr uint64_t kQPlanes = (1ull << kQP) - 1ull;

// One cell's state. Its size is 8 words modulo 32, so that the four groups'
// equal offsets fall on different banks.
struct __align__(16) QuadCell {
  float4 vp[kQV];      // position, error bound; with pl the scratch of the FP64 integration
  float4 pl[kQP];      // n^, b^
  float pe[kQP];       // offset error bound; the FP64 integration's face anchors
  int pid[kQP];        // sorted site index, or -1-f for box face f
  uint32_t vt[kQV];    // plane triplet
  uint32_t otri[kQV];  // triplets a clip removes (bits 24 up: their slots); the neighbour list
  unsigned short edge[kQV];  // edges of a clip's hole; slots to fill
  float4 cpl[kQC];     // candidate planes, their bounds and sites
  float ce[kQC];
  int cid[kQC];
  int knn[kKnn];
  unsigned tally[8];  // of the group's finished cells: FP64 signs, those still ambiguous, vertices and volumes re-solved,
                      // empty cells
};
static_assert(sizeof(QuadCell) % 128 == 32, "bank layout");
struct __align__(16) QuadWarp {
  QuadCell cell[4];
  uint32_t qkey[kQQ];  // ordered key (17 bits), children to visit (8), free for the slot (7)
  int qref[kQQ];       // inner node, and the groups that want it from bit 26 up
};
static_assert(kQF * kQF <= kQC * (16 + 4 + 4), "edge table over the candidate arrays");
static_assert(kKnn == 8, "one KNN site per lane of a group");
static_assert(sizeof(double) * 3 * kQV <= sizeof(float4) * (kQV + kQP), "FP64 scratch");

enum { T_SIGNS = 0, T_AMB = 1, T_VERTS = 2, T_VOLS = 3, T_EMPTY = 4, T_COUNT = 5 };
enum { M_BUILD = 0, M_EMPTY = 1, M_OVERFLOW = 2, M_IDLE = 3 };

// reductions over the 8 lanes of a group
__device__ __forceinline__ float group_min(float v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(FULL, v, o));
  return v;
}
__device__ __forceinline__ float group_max(float v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
  return v;
}
__device__ __forceinline__ uint32_t group_minu(uint32_t v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(FULL, v, o));
  return v;
}
__device__ __forceinline__ uint32_t group_or(uint32_t v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v |= __shfl_xor_sync(FULL, v, o);
  return v;
}
__device__ __forceinline__ int group_add(int v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}

__device__ __forceinline__ PlaneT<float> quad_plane(const QuadCell& S, int k) {
  const float4 t = S.pl[k];
  PlaneT<float> P;
  P.nx = t.x;
  P.ny = t.y;
  P.nz = t.z;
  P.b = t.w;
  P.e = S.pe[k];
  return P;
}

// Volume and first moment about (cx, cy, cz) in FP64 of the groups with
// nv > 0 (the scheme of volume_fp64: vertices re-solved from the inputs, each
// face's fan anchored at its lowest vertex). Overwrites vp, pl and pe.
__device__ __noinline__ void quad_volume64(QuadCell& S, int nv, float4 me, const float* box,
                                           const float4* __restrict__ sites, double cx, double cy, double cz,
                                           double& V, double& Mx, double& My, double& Mz) {
  const int gl = (int)(lane_id() & 7u);
  double* vd64 = reinterpret_cast<double*>(S.vp);
  int* anchor = reinterpret_cast<int*>(S.pe);
  if (nv > 0)
    for (int f = gl; f < kQP; f += 8) anchor[f] = 0x7fffffff;
  __syncwarp();
#pragma unroll 1
  for (int t = gl; t < nv; t += 8) {
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
  V = Mx = My = Mz = 0.0;
#pragma unroll 1
  for (int it = gl; it < 3 * nv; it += 8) {
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
  V = group_sum(V) / 6.0;
  Mx = group_sum(Mx) / 24.0;
  My = group_sum(My) / 24.0;
  Mz = group_sum(Mz) / 24.0;
}

// The tape record (see write_tape in vd_cells.cu) of the groups with `on`;
// otri holds the renumbered triplets.
__device__ __noinline__ void quad_tape(const QuadCell& S, char* rec, int nv, int nf, uint64_t alive, bool on) {
  const int gl = (int)(lane_id() & 7u);
  if (!on) return;
  const bool fits = nv <= kTapeV && nf <= kTapeF;
  if (fits) {
    float4* tv = reinterpret_cast<float4*>(rec + kTapeVOff);
#pragma unroll 1
    for (int t = gl; t < nv; t += 8) {
      const float4 p = S.vp[t];
      tv[t] = make_float4(p.x, p.y, p.z, __uint_as_float(S.otri[t]));
    }
    int* tf = reinterpret_cast<int*>(rec + kTapeFOff);
#pragma unroll 1
    for (int f = gl; f < kQP; f += 8)
      if ((alive >> f) & 1ull) tf[__popcll(alive & ((1ull << f) - 1ull))] = S.pid[f];
  }
  if (gl == 0) *reinterpret_cast<int4*>(rec) = make_int4(fits ? nv : -1, nf, 0, 0);
}

__global__ void __launch_bounds__(128, 4) quad_kernel(CellBuffers P) {
  extern __shared__ __align__(16) unsigned char quad_smem[];
  const unsigned lane = lane_id();
  const int gl = (int)(lane & 7u);
  const unsigned gsh = lane & 24u;
  const uint32_t ltg = (1u << gl) - 1u;
  QuadWarp& W = reinterpret_cast<QuadWarp*>(quad_smem)[threadIdx.x >> 5];
  QuadCell& S = W.cell[lane >> 3];
  auto group_ballot = [&](bool p) { return (__ballot_sync(FULL, p) >> gsh) & 255u; };
  const float u = Num<float>::u;
  S.tally[gl] = 0;

  while (true) {
    int item = 0;
    if (lane == 0) item = atomicAdd(&P.work[0], 4);
    // always the same four cells: the order in which a cell meets its planes,
    // hence its last bits, hang on the other three. A part of a diagram makes
    // all four where its range ends between them, and writes its own
    item = (P.cell_begin & ~3) + __shfl_sync(FULL, item, 0);
    if (item >= P.cell_end) break;
    const bool exists = item + (int)(lane >> 3) < P.n;
    const int si = exists ? item + (int)(lane >> 3) : item;
    const bool own = exists && si >= P.cell_begin && si < P.cell_end;
    const float4 me = P.sites[si];
    const int orig = P.perm[si];
    const SetInfo& SI = P.sets[P.nsets > 1 ? (int)(P.keys[si] >> P.set_shift) : 0];
    const float* box = SI.lo;
    // a site that an exact duplicate beats has an empty cell
    int mode = !exists ? M_IDLE : (P.loser[si] || !finite_site(me) ? M_EMPTY : M_BUILD);
    unsigned ct64 = 0, ctamb = 0, ctrefv = 0;  // this cell's, a lane's share

    // ---- the box: 6 planes, 8 corners (as init_cell)
    if (gl < 6) {
      const PlaneT<float> B = box_plane<float>(gl, me.x, me.y, me.z, box, box + 3);
      S.pl[gl] = make_float4(B.nx, B.ny, B.nz, B.b);
      S.pe[gl] = B.e;
      S.pid[gl] = -1 - gl;
    }
    __syncwarp();
    {
      const int sx = gl & 1, sy = (gl >> 1) & 1, sz = gl >> 2;
      const bool odd = (sx + sy + sz) & 1;
      const uint32_t b = odd ? 4 + sz : 2 + sy, d = odd ? 2 + sy : 4 + sz;
      const float px = S.pl[sx].w, py = S.pl[2 + sy].w, pz = S.pl[4 + sz].w;
      const float x = sx ? -px : px, y = sy ? -py : py, z = sz ? -pz : pz;
      const float x1 = fabsf(x) + fabsf(y) + fabsf(z);
      const float ep = 1.75f * (S.pe[sx] + S.pe[2 + sy] + S.pe[4 + sz]) + (5.25f * 8.0f * u + 9.0f * u) * x1 +
                       6.0f * u * x1 + u * x1;
      S.vp[gl] = make_float4(x, y, z, x1 < 1e30f ? 1.1f * ep + 11.0f * u * x1 : INFINITY);
      S.vt[gl] = (uint32_t)sx | (b << 8) | (d << 16);
    }
    int nv = mode == M_BUILD ? 8 : 0;
    uint64_t freem = kQPlanes & ~63ull;
    // ---- the walk starts at the roots of the cells' sets (one, except where
    // sets meet); before it, each cell is clipped by its KNN list, which makes
    // the bounds tight from the first node test on (without it, or from a
    // window of the sorted order instead, the walk visits twice the nodes)
    int qn = 0;
    int visits = 0;  // nodes visited
    int cur = -1;  // the node to visit next (as in qref), if it is not the queue's best
    {
      const unsigned same = __match_any_sync(FULL, SI.first);
      const bool head = (same & lanemask_lt()) == 0;
      const unsigned heads = __ballot_sync(FULL, head);
      qn = __popc(heads);
      if (head) {
        const int at = __popc(heads & lanemask_lt());
        const unsigned gm = (same & 1u) | ((same >> 7) & 2u) | ((same >> 14) & 4u) | ((same >> 21) & 8u);
        W.qkey[at] = 255u << 7;
        W.qref[at] = (int)((gm << 26) | (unsigned)(ref_is_leaf(SI.wroot) ? kQLeafRoot : SI.wroot));
      }
    }
    S.knn[gl] = P.knn[(size_t)si * kKnn + gl];
    int cn = 0, cf = 0;  // candidates, those with a plane already
    bool knn_turn = true;
    uint32_t pend = 0;  // bit 8 g + c: cell g has yet to read child c, a leaf, of the node visited last
    int cref = 0;       // reference of that node's child gl
    __syncwarp();

    bool dirty = true;
    WalkBounds B;
    const bool weighted = __any_sync(FULL, SI.weighted != 0);

#pragma unroll 1
    while (true) {
      // ---- A: bounds of the polytopes
      if (__any_sync(FULL, dirty)) {
        float mn0 = INFINITY, mn1 = INFINITY, mn2 = INFINITY, mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY;
        float em = 0.f;
#pragma unroll 1
        for (int v = gl; v < nv; v += 8) {
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
        em = group_max(em);
        B.lo[0] = group_min(mn0) - em;
        B.lo[1] = group_min(mn1) - em;
        B.lo[2] = group_min(mn2) - em;
        B.hi[0] = group_max(mx0) + em;
        B.hi[1] = group_max(mx1) + em;
        B.hi[2] = group_max(mx2) + em;
#pragma unroll
        for (int k = 0; k < 3; k++) {
          B.lo2[k] = B.lo[k] * B.lo[k];
          B.hi2[k] = B.hi[k] * B.hi[k];
          B.c[k] = 0.5f * (B.lo[k] + B.hi[k]);
        }
        float r2 = 0.f;
#pragma unroll 1
        for (int v = gl; v < nv; v += 8) {
          const float4 p = S.vp[v];
          const float dx = p.x - B.c[0], dy = p.y - B.c[1], dz = p.z - B.c[2];
          r2 = fmaxf(r2, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        }
        __syncwarp();
        B.rad = (sqrt_approx(group_max(r2)) + em) * (1.0f + kCullPad);
        const float reach = sqrt_approx(B.c[0] * B.c[0] + B.c[1] * B.c[1] + B.c[2] * B.c[2]) + B.rad;
        B.reach2 = reach * reach;
        B.ext = 4.0f * (reach + fabsf(B.c[0]) + fabsf(B.c[1]) + fabsf(B.c[2]) + B.rad);
        dirty = false;
      }

      // ---- T: walk until a cell's list is nearly full or nothing is left
      bool finished = false, clip_now = false;
#pragma unroll 1
      while (!__any_sync(FULL, cn > kQT)) {
        if (!knn_turn && pend == 0) {
          if (qn == 0 && cur < 0) {
            finished = clip_now = true;
            break;
          }
          if (++visits > kQN) {
            if (mode == M_BUILD) mode = M_OVERFLOW;
            cn = 0;
            qn = 0;
            cur = -1;
            continue;
          }
          // visit the best node: its 8 children, one per lane of each group
          uint32_t todo = 255u;
          int e = cur;
          if (cur < 0) {
            uint32_t best = 0xffffffffu;
            for (int q = (int)lane; q < qn; q += 32) best = min(best, W.qkey[q] | (uint32_t)q);
            best = __reduce_min_sync(FULL, best);
            const int at = (int)(best & 127u);
            todo = (best >> 7) & 255u;
            e = W.qref[at];
            qn--;
            __syncwarp();
            if (lane == 0) {
              W.qkey[at] = W.qkey[qn];
              W.qref[at] = W.qref[qn];
            }
            __syncwarp();
          }
          cur = -1;
          const int node = e & ((1 << 26) - 1);
          const bool act = mode == M_BUILD && ((e >> (26 + (lane >> 3))) & 1);
          bool keep = false;
          float key = 0.f;
          if (node == kQLeafRoot) {  // sets of one leaf (each group its own)
            cref = SI.wroot;
            keep = act && gl == 0;
          } else {
            const float4* nd = P.wide + 16 * (size_t)node + gl;
            const float4 lo = __ldg(nd), hi = __ldg(nd + 8);
            cref = __float_as_int(hi.w);
            float lb;
            keep = walk_node_test(lo, hi, me, B, weighted, key, lb) && act && ((todo >> gl) & 1u) && cref != kNoChild;
          }
          pend = __ballot_sync(FULL, keep && ref_is_leaf(cref));
          const uint32_t inner = __ballot_sync(FULL, keep && !ref_is_leaf(cref));
          if (inner) {
            uint32_t kk = (inner >> lane) & 1u ? f2o(key) : 0xffffffffu;
            kk = min(kk, __shfl_xor_sync(FULL, kk, 8));
            kk = min(kk, __shfl_xor_sync(FULL, kk, 16));
            const uint32_t any = (inner | (inner >> 8) | (inner >> 16) | (inner >> 24)) & 255u;
            const uint32_t t = inner >> gl;
            const int child = (int)((((t & 1u) | ((t >> 7) & 2u) | ((t >> 14) & 4u) | ((t >> 21) & 8u)) << 26) | (unsigned)cref);
            if (qn + __popc(any) > kQQ - 24) {
              // little room (bounds still loose in several directions): go on
              // with the best child, and queue the node itself with the
              // others, to be tested again under the bounds of that time
              const uint32_t b1 = __reduce_min_sync(FULL, (any >> gl) & 1u ? ((kk & ~7u) | (uint32_t)gl) : 0xffffffffu);
              const int src = (int)(b1 & 7u);
              const uint32_t rest = any & ~(1u << src);
              cur = __shfl_sync(FULL, child, src);
              if (rest) {
                const uint32_t b2 = __reduce_min_sync(FULL, (rest >> gl) & 1u ? kk : 0xffffffffu);
                if (qn >= kQQ) {  // no room at all: cells that reach far into the tree
                  if (mode == M_BUILD) mode = M_OVERFLOW;
                  cn = 0;
                  qn = 0;
                  pend = 0;
                  cur = -1;
                  continue;
                }
                if (lane == 0) {
                  W.qkey[qn] = (b2 & ~0x7fffu) | (rest << 7);
                  W.qref[qn] = e;
                }
                qn++;
                __syncwarp();
              }
              continue;
            }
            if (lane < 8 && ((any >> lane) & 1u)) {
              const int to = qn + __popc(any & ltg);
              W.qkey[to] = (kk & ~0x7fffu) | (255u << 7);
              W.qref[to] = child;
            }
            qn += __popc(any);
            __syncwarp();
          }
          continue;
        }
        // read a leaf (or the KNN lists): two sites per lane, for the cells
        // that want it. Losers of a duplicate position and sites clipped before
        // are sorted out later, where the candidates stand close together
        int j0 = S.knn[gl], lim = j0;
        bool want = mode == M_BUILD;
        if (!knn_turn) {
          const uint32_t any = pend | (pend >> 8) | (pend >> 16) | (pend >> 24);
          const int c = __ffs(any) - 1;  // a leaf root is child 0 of each group of its own
          const int ref = __shfl_sync(FULL, cref, c, 8);
          j0 = leaf_first(ref) + gl;
          lim = leaf_first(ref) + leaf_count(ref) - 1;
          want = want && ((pend >> (gsh + c)) & 1u);
          pend &= ~(0x01010101u << c);
        }
        float4 q[2];
        bool act[2], keep[2];
#pragma unroll
        for (int r = 0; r < 2; r++) {
          const int j = j0 + 8 * r;
          act[r] = want & (j >= 0) & (j <= lim) & (j != si);
          q[r] = P.sites[act[r] ? j : si];
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
              lose = lose || q[r].w > me.w || (q[r].w == me.w && P.perm[j0 + 8 * r] < orig);
            }
          if (group_ballot(lose)) mode = M_EMPTY;
        }
#pragma unroll
        for (int r = 0; r < 2; r++) {
          const uint32_t km = group_ballot(keep[r]);
          if (keep[r]) {
            const int at = cn + __popc(km & ltg);
            S.cpl[at] = q[r];
            S.cid[at] = j0 + 8 * r;
          }
          cn += __popc(km);
        }
        if (mode != M_BUILD) cn = 0;
        if (knn_turn) {
          clip_now = true;
          break;
        }
      }
      __syncwarp();
      // the candidates' planes, eight at a time (a leaf step finds one or two
      // per cell)
#pragma unroll 1
      for (int q = cf + gl; q < cn; q += 8) {
        const float4 p = S.cpl[q];
        const int id = S.cid[q];
        PlaneT<float> c = site_plane<float>(me.x, me.y, me.z, me.w, p.x, p.y, p.z, p.w);
        bool drop = P.loser[id] != 0;
        if (!knn_turn) {
          const int4 a = *reinterpret_cast<const int4*>(&S.knn[0]), b = *reinterpret_cast<const int4*>(&S.knn[4]);
          drop = drop | (id == a.x) | (id == a.y) | (id == a.z) | (id == a.w) | (id == b.x) | (id == b.y) | (id == b.z) |
                 (id == b.w);
        }
        S.cpl[q] = make_float4(c.nx, c.ny, c.nz, drop ? INFINITY : c.b);  // F drops what cuts nothing
        S.ce[q] = drop ? 0.f : c.e;
      }
      knn_turn = false;
      __syncwarp();

#pragma unroll 1
      while (true) {
        // ---- F: candidates that leave every vertex inside are dropped for good
        // (clipping only shrinks the cell); the nearest of the others is next
        uint32_t key = 0xffffffffu;
        {
          int kept = 0;
#pragma unroll 1
          for (int base = 0; __any_sync(FULL, base < cn); base += 8) {
            const int q = base + gl;
            bool any = false;
            float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
            float he = 0.f;
            int id = 0;
            if (q < cn) {
              h = S.cpl[q];
              he = S.ce[q];
              id = S.cid[q];
              // the sign test's value plus both error bounds (a little more of
              // each than the classification takes), as one chain per vertex
              const float nb = fmaf(1.25f, he, -h.w);
              float top = -INFINITY;
#pragma unroll 4
              for (int v = 0; v < nv; v++) {
                const float4 p = S.vp[v];
                top = fmaxf(top, fmaf(h.x, p.x, fmaf(h.y, p.y, fmaf(h.z, p.z, fmaf(1.0001f, p.w, nb)))));
              }
              any = top > 0.f;
            }
            __syncwarp();
            const uint32_t km = group_ballot(any);
            const int to = kept + __popc(km & ltg);
            if (any) {
              if (to != q) {
                S.cpl[to] = h;
                S.ce[to] = he;
                S.cid[to] = id;
              }
              key = min(key, (f2o(h.w) & ~31u) | (uint32_t)to);
            }
            kept += __popc(km);
            __syncwarp();
          }
          cn = kept;
        }
        const bool act = cn > 0;
        if (!(clip_now ? __any_sync(FULL, act) : __any_sync(FULL, cn > kQS))) break;
        clip_now = true;
        // ---- C: classify the vertices
        PlaneT<float> H;
        H.nx = H.ny = H.nz = H.b = H.e = 0.f;
        int hj = 0, k = 0;
        uint32_t outm = 0;  // bit s: vertex 8 s + gl lies outside
        bool cut = false;
        {
          key = group_minu(key);
          if (act) {
            const int at = (int)(key & 31u);
            const float4 p = S.cpl[at];
            H.nx = p.x;
            H.ny = p.y;
            H.nz = p.z;
            H.b = p.w;
            H.e = S.ce[at];
            hj = S.cid[at];
          }
          __syncwarp();
          if (act) {  // the last candidate takes its place
            const int at = (int)(key & 31u);
            cn--;
            if (gl == 0) {
              S.cpl[at] = S.cpl[cn];
              S.ce[at] = S.ce[cn];
              S.cid[at] = S.cid[cn];
            }
          }
          uint32_t ambm = 0;
          if (act) {
            uint32_t bit = 1;
#pragma unroll 1
            for (int v = gl; v < nv; v += 8, bit <<= 1) {
              const float4 p = S.vp[v];
              const float s = side<float>(H, p.x, p.y, p.z);
              if (ambiguous<float>(s, p.w, H.e))
                ambm |= bit;
              else if (s > 0.0f)
                outm |= bit;
            }
          }
          __syncwarp();
          if (__any_sync(FULL, ambm != 0)) {
            while (ambm) {
              const int s = __ffs(ambm) - 1;
              ambm &= ambm - 1;
              ct64++;
              const unsigned r = walk_resolve64(S.pid, S.vt[8 * s + gl], hj, me, box, P.sites);
              outm |= (r & 1u) << s;
              ctamb += r >> 1;
            }
            __syncwarp();
          }
          const int kk = group_add(__popc(outm));
          if (act && kk > 0) {
            k = kk;
            if (k == nv) {
              mode = M_EMPTY;
              cn = 0;
            } else {
              cut = true;
            }
          }
        }

        // ---- H: clip by the plane found (App. B)
        if (!__any_sync(FULL, cut)) continue;
        // a plane slot for it; slots that no kept vertex uses are reclaimed when none is free
        if (__any_sync(FULL, cut && freem == 0)) {
          uint32_t lo = 0, hi = 0;
          if (cut) {
            uint32_t bits = outm;
            for (int v = gl; v < nv; v += 8, bits >>= 1) {
              if (bits & 1u) continue;
              const uint32_t T = S.vt[v];
#pragma unroll
              for (int c = 0; c < 3; c++) {
                const uint32_t f = (T >> (8 * c)) & 255u;
                if (f < 32u)
                  lo |= 1u << f;
                else
                  hi |= 1u << (f - 32u);
              }
            }
          }
          __syncwarp();
          lo = group_or(lo);
          hi = group_or(hi);
          if (cut && freem == 0) freem = kQPlanes & ~(((uint64_t)hi << 32) | lo);
          if (cut && freem == 0) {
            mode = M_OVERFLOW;
            cut = false;
            cn = 0;
          }
        }
        int h = 0;
        if (cut) {
          h = __ffsll((long long)freem) - 1;
          freem &= freem - 1;
          if (gl == 0) {
            S.pl[h] = make_float4(H.nx, H.ny, H.nz, H.b);
            S.pe[h] = H.e;
            S.pid[h] = hj;
          }
        }
        // the removed vertices' triplets and slots
        int gone;
        {
          const int c = cut ? __popc(outm) : 0;
          int before = c;
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) {
            const int t = __shfl_up_sync(FULL, before, o, 8);
            if (gl >= o) before += t;
          }
          before -= c;
          if (cut)
            for (uint32_t bits = outm; bits; bits &= bits - 1) {
              const int v = 8 * (__ffs(bits) - 1) + gl;
              S.otri[before++] = S.vt[v] | ((uint32_t)v << 24);
            }
          gone = k;
        }
        __syncwarp();
        // the hole's edges: every directed pair (a, b) of a removed vertex whose
        // reverse is in no other removed vertex -> vertex (a, b, h). One removed
        // vertex per lane
        int m = 0;
        {
          const int kmax = __reduce_max_sync(FULL, cut ? k : 0);
#pragma unroll 1
          for (int base = 0; base < kmax; base += 8) {
            const int t = base + gl;
            const bool own = cut && t < k;
            const uint32_t T = own ? S.otri[t] : 0u;
            const uint32_t a = T & 255u, b = (T >> 8) & 255u, c = (T >> 16) & 255u;
            const uint32_t r0 = b | (a << 8), r1 = c | (b << 8), r2 = a | (c << 8);
            bool e0 = own, e1 = own, e2 = own;
#pragma unroll 1
            for (int v = 0; v < kmax; v++) {
              const uint32_t U = v < k ? S.otri[v] : 0u;
              const uint32_t p0 = U & 0xffffu, p1 = (U >> 8) & 0xffffu, p2 = ((U >> 16) & 255u) | ((U & 255u) << 8);
              e0 = e0 && p0 != r0 && p1 != r0 && p2 != r0;
              e1 = e1 && p0 != r1 && p1 != r1 && p2 != r1;
              e2 = e2 && p0 != r2 && p1 != r2 && p2 != r2;
            }
            const uint32_t m0 = group_ballot(e0), m1 = group_ballot(e1), m2 = group_ballot(e2);
            int at = m + __popc(m0 & ltg) + __popc(m1 & ltg) + __popc(m2 & ltg);
            if (e0 && at < kQV) S.edge[at] = (unsigned short)(a | (b << 8));
            at += e0;
            if (e1 && at < kQV) S.edge[at] = (unsigned short)(b | (c << 8));
            at += e1;
            if (e2 && at < kQV) S.edge[at] = (unsigned short)(c | (a << 8));
            m += __popc(m0) + __popc(m1) + __popc(m2);
          }
        }
        if (cut && nv - gone + m > kQV) {
          mode = M_OVERFLOW;
          cut = false;
          cn = 0;
        }
        __syncwarp();
        // new vertex t takes the slot of removed vertex t, then slots at the end
#pragma unroll 1
        for (int base = 0; __any_sync(FULL, cut && base < m); base += 8) {
          const int t = base + gl;
          if (cut && t < m) {
            const uint32_t ab = S.edge[t];
            const int a = (int)(ab & 255u), b = (int)(ab >> 8);
            const int at = t < gone ? (int)(S.otri[t] >> 24) : nv + (t - gone);
            float x, y, z, ev;
            vertex3<float>(quad_plane(S, a), quad_plane(S, b), H, x, y, z, ev);
            S.vp[at] = make_float4(x, y, z, ev);
            S.vt[at] = ab | ((uint32_t)h << 16);
            if (!(ev <= kRefineRel * (fabsf(x) + fabsf(y) + fabsf(z)))) {
              walk_refine(&S.vp[at], S.pid[a], S.pid[b], hj, me, box, P.sites);
              ctrefv++;
            }
          }
        }
        __syncwarp();
        // fewer new vertices than removed ones: the slots left over are filled
        // from the end of the array
        if (__any_sync(FULL, cut && m < gone)) {
          const int left = cut ? max(gone - m, 0) : 0, to = nv - left;
          for (int t = gl; t < left; t += 8) S.vt[S.otri[m + t] >> 24] = kEmptyTri;
          __syncwarp();
          int holes = 0, live = 0;
          const int lmax = __reduce_max_sync(FULL, left);
#pragma unroll 1
          for (int base = 0; base < lmax; base += 8) {
            const int t = base + gl;
            const int slot = t < left ? (int)(S.otri[m + t] >> 24) : kQV;
            const uint32_t hm = group_ballot(slot < to);
            if (slot < to) S.edge[holes + __popc(hm & ltg)] = (unsigned short)slot;
            holes += __popc(hm);
          }
          __syncwarp();
#pragma unroll 1
          for (int base = 0; base < lmax; base += 8) {
            const int v = to + base + gl;
            const bool mv = base + gl < left && S.vt[v] != kEmptyTri;
            const uint32_t vm = group_ballot(mv);
            if (mv) {
              const int slot = (int)S.edge[live + __popc(vm & ltg)];
              S.vp[slot] = S.vp[v];
              S.vt[slot] = S.vt[v];
            }
            live += __popc(vm);
          }
          __syncwarp();
        }
        if (cut) {
          nv += m - gone;
          dirty = true;
        }
      }
      cf = cn;
      if (finished || !__any_sync(FULL, mode == M_BUILD)) break;
    }

    // ---- outputs
    if (!own) mode = M_IDLE;
    if (mode == M_EMPTY) {
      if (gl == 0) {
        atomicAdd(&S.tally[T_EMPTY], 1u);
        P.counts[orig] = 0;
        P.vol[orig] = 0.0f;
        P.cen[3 * (size_t)orig] = me.x;
        P.cen[3 * (size_t)orig + 1] = me.y;
        P.cen[3 * (size_t)orig + 2] = me.z;
      }
    }
    if (mode == M_OVERFLOW && gl == 0) {  // to the one-cell-per-warp kernel
      P.mid_list[atomicAdd(&P.st->mid_count, 1)] = si;
      if (P.tape) *reinterpret_cast<int4*>(P.tape + (size_t)si * kTapeStride) = make_int4(-1, 0, 0, 0);
    }
    const bool done = mode == M_BUILD;
    if (!done) nv = 0;
    if (__any_sync(FULL, done)) {
      float sx = 0.f, sy = 0.f, sz = 0.f, emax = 0.f;
      uint32_t lom = 0, him = 0;
#pragma unroll 1
      for (int v = gl; v < nv; v += 8) {
        const float4 p = S.vp[v];
        const uint32_t T = S.vt[v];
        sx += p.x;
        sy += p.y;
        sz += p.z;
        emax = fmaxf(emax, p.w);
#pragma unroll
        for (int c = 0; c < 3; c++) {
          const uint32_t f = (T >> (8 * c)) & 255u;
          if (f < 32u)
            lom |= 1u << f;
          else
            him |= 1u << (f - 32u);
        }
      }
      __syncwarp();
      const uint64_t alive = ((uint64_t)group_or(him) << 32) | group_or(lom);
      sx = group_sum(sx);
      sy = group_sum(sy);
      sz = group_sum(sz);
      emax = group_max(emax);
      // neighbours: site planes that carry a face, ascending
      int nb = 0;
#pragma unroll 1
      for (int f = gl; f < kQP; f += 8) {
        const bool isn = done && ((alive >> f) & 1ull) && S.pid[f] >= 0;
        const uint32_t mk = group_ballot(isn);
        if (isn) S.otri[nb + __popc(mk & ltg)] = (uint32_t)(P.perm[S.pid[f]] - SI.first);
        nb += __popc(mk);
      }
      __syncwarp();
      int* row = P.scratch + (size_t)orig * P.stride;
#pragma unroll 1
      for (int t = gl; t < nb; t += 8) {
        const int v = (int)S.otri[t];
        int rank = 0;
#pragma unroll 4
        for (int w = 0; w < nb; w++) rank += (int)S.otri[w] < v;
        row[rank] = v;
      }
      __syncwarp();
      // triplets in the order of the planes that carry a face (otri), and the
      // vertex that each directed plane pair belongs to (succ), so that an
      // edge's other end is one look-up (a search took 25 steps for the
      // slowest lane, most of this stage's time)
      const int nf = __popcll(alive);
      unsigned char* succ = reinterpret_cast<unsigned char*>(S.cpl);
      const bool direct = nf <= kQF;
#pragma unroll 1
      for (int v = gl; v < nv; v += 8) {
        const uint32_t T = S.vt[v];
        uint32_t R = 0;
#pragma unroll
        for (int c = 0; c < 3; c++) {
          const uint32_t f = (T >> (8 * c)) & 255u;
          R |= (uint32_t)__popcll(alive & ((1ull << f) - 1ull)) << (8 * c);
        }
        S.otri[v] = R;
        if (direct) {
          const uint32_t a = R & 255u, b = (R >> 8) & 255u, c = R >> 16;
          succ[a * kQF + b] = (unsigned char)v;
          succ[b * kQF + c] = (unsigned char)v;
          succ[c * kQF + a] = (unsigned char)v;
        }
      }
      __syncwarp();
      if (P.tape) quad_tape(S, P.tape + (size_t)si * kTapeStride, nv, nf, alive, done);
      // volume and first moment: tetrahedra (c, g_f, v, w) as in cell_outputs
      const float inv = 1.0f / (float)max(nv, 1);
      const float cx = sx * inv, cy = sy * inv, cz = sz * inv;
      float V = 0.f, Mx = 0.f, My = 0.f, Mz = 0.f, Sabs = 0.f;
#pragma unroll 1
      for (int it = gl; it < 3 * nv; it += 8) {
        const int t = it / 3, rho = it - 3 * t;
        const uint32_t T = S.vt[t], R = S.otri[t];
        const uint32_t fy = ((T | (T << 24)) >> (8 * rho + 8)) & 255u;
        const uint32_t xy = ((R | (R << 24)) >> (8 * rho)) & 0xffffu, x = xy & 255u, y = xy >> 8;
        int w = 0;
        if (direct)
          w = succ[y * kQF + x];
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
      V = group_sum(V) * (1.0f / 6.0f);
      Mx = group_sum(Mx) * (1.0f / 24.0f);
      My = group_sum(My) * (1.0f / 24.0f);
      Mz = group_sum(Mz) * (1.0f / 24.0f);
      Sabs = group_sum(Sabs) * 0.5f;
      float L = 0.f;
#pragma unroll
      for (int c = 0; c < 3; c++) L += fmaxf(B.lo2[c], B.hi2[c]);
      L = sqrtf(L);
      double ox = cx, oy = cy, oz = cz, Vd = V;
      const bool need64 = done && volume_needs_fp64(V, L, Sabs, emax);
      if (__any_sync(FULL, need64)) {
        double V6, X6, Y6, Z6;
        quad_volume64(S, need64 ? nv : 0, me, box, P.sites, (double)cx, (double)cy, (double)cz, V6, X6, Y6, Z6);
        if (need64) {
          Vd = V6;
          if (V6 > 0.0) {
            const double iv = 1.0 / V6;
            ox += X6 * iv;
            oy += Y6 * iv;
            oz += Z6 * iv;
          }
          if (gl == 0) atomicAdd(&S.tally[T_VOLS], 1u);
        }
      }
      if (!need64 && V > 0.0f) {
        ox += Mx / V;
        oy += My / V;
        oz += Mz / V;
      }
      if (done && gl == 0) {
        P.counts[orig] = nb;
        P.vol[orig] = (float)Vd;
        P.cen[3 * (size_t)orig] = (float)((double)me.x + ox);
        P.cen[3 * (size_t)orig + 1] = (float)((double)me.y + oy);
        P.cen[3 * (size_t)orig + 2] = (float)((double)me.z + oz);
      }
    }
    // the events of cells that this kernel finishes: of one passed on, the next
    // kernel counts them, of a neighbouring part's cell, that part's build
    const bool kept = mode == M_BUILD || mode == M_EMPTY;
    const uint32_t am = group_ballot(kept && ctamb != 0);
    if (am && gl == 0) record_ambiguous(P.st, P.amb_list, P.amb_cap, orig);
    if (kept && ctrefv) atomicAdd(&S.tally[T_VERTS], ctrefv);
    if (kept && ct64) {
      atomicAdd(&S.tally[T_SIGNS], ct64);
      atomicAdd(&S.tally[T_AMB], ctamb);
    }
    __syncwarp();
  }
  __syncwarp();
  unsigned sum = S.tally[gl];
  sum += __shfl_xor_sync(FULL, sum, 8);
  sum += __shfl_xor_sync(FULL, sum, 16);
  if (lane < T_COUNT && sum) {
    long long* to = lane == T_SIGNS   ? &P.st->fp64_fallbacks
                    : lane == T_AMB   ? &P.st->fp64_ambiguous
                    : lane == T_VERTS ? &P.st->refined_vertices
                    : lane == T_VOLS  ? &P.st->refined_volumes
                                      : &P.st->empty_cells;
    atomicAdd((unsigned long long*)to, (unsigned long long)sum);
  }
}

}  // namespace

cudaError_t launch_quad(const CellBuffers& c, int num_sms, cudaStream_t s) {
  const int wpb = c.cfg.warps_per_block > 4 ? 4 : c.cfg.warps_per_block;
  const size_t smem = sizeof(QuadWarp) * (size_t)wpb;
  cudaError_t err = cudaFuncSetAttribute(quad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  int per_sm = c.cfg.blocks_per_sm;
  if (per_sm <= 0) {
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, quad_kernel, 32 * wpb, smem);
    if (err != cudaSuccess) return err;
    if (per_sm <= 0) per_sm = 1;
  }
  const int m = c.cell_end - (c.cell_begin & ~3);
  int blocks = (m + 4 * wpb - 1) / (4 * wpb);
  blocks = blocks < 1 ? 1 : (blocks < num_sms * per_sm ? blocks : num_sms * per_sm);
  quad_kernel<<<blocks, 32 * wpb, smem, s>>>(c);
  return cudaGetLastError();
}

}  // namespace vd
