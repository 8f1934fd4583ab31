// vd_bvh.cu -- input packing, Morton keys, radix sort and the power-augmented
// LBVH (App. A.1 "Input packing", App. A.2 "Power-augmented BVH"; the paper
// uses a third-party builder, this is a Karras-style binary radix tree over
// Morton-sorted sites, collapsed to leaves of at most `leaf_size` sites, with
// a per-node maximum weight for the culling test of Sec. 4.2.2).
#include <algorithm>
#include <utility>

#include "vd_internal.cuh"

namespace vd {

// ---------------------------------------------------------------- Morton keys

__device__ __forceinline__ uint64_t spread3(uint32_t v) {
  // spread the low 21 bits of v so that bit k lands on bit 3k (callers use
  // at most 20 bits per axis)
  uint64_t x = v & 0x1fffffu;
  x = (x | (x << 32)) & 0x1f00000000ffffull;
  x = (x | (x << 16)) & 0x1f0000ff0000ffull;
  x = (x | (x << 8)) & 0x100f00f00f00f00full;
  x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
  x = (x | (x << 2)) & 0x1249249249249249ull;
  return x;
}

__host__ __device__ __forceinline__ int find_set(const SetInfo* sets, int nsets, int i) {
  int lo = 0, hi = nsets - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (sets[mid].first <= i)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// Range of the weights of weighted sets: wr[0] the complement of the least
// orderable value, wr[1] the greatest, so that both start at 0 (no weight).
__global__ void weight_range_kernel(const float* __restrict__ w, int n, const SetInfo* __restrict__ sets, int nsets,
                                    unsigned* __restrict__ wr) {
  uint32_t mn = 0xffffffffu, mx = 0u;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int s = nsets > 1 ? find_set(sets, nsets, i) : 0;
    if (!sets[s].weighted || !isfinite(w[i])) continue;
    uint32_t o = f2o(w[i]);
    mn = min(mn, o);
    mx = max(mx, o);
  }
  mn = __reduce_min_sync(FULL, mn);
  mx = __reduce_max_sync(FULL, mx);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&wr[0], ~mn);
    atomicMax(&wr[1], mx);
  }
}

cudaError_t launch_weight_range(const float* w, int n, const SetInfo* sets, int nsets, unsigned* wr,
                                cudaStream_t s) {
  if (!w) return cudaGetLastError();
  int blocks = min((n + 255) / 256, 1024);
  weight_range_kernel<<<blocks, 256, 0, s>>>(w, n, sets, nsets, wr);
  return cudaGetLastError();
}

// Weight stratum of a site (a performance device only; any partition
// gives the same cells): with o = w - w_min and O = w_max - w_min, bin 7
// holds o in (O/4, O], bin 6 (O/16, O/4], ... bin 0 everything below.
// Sorting by (bin, Morton) puts each stratum in its own subtrees, so a
// node's maximum weight -- the w_max of the node bound of Sec. 4.2.2 --
// is within a factor 4 of its sites' weights instead of the global maximum.
__device__ __forceinline__ uint32_t weight_bin(float w, float wmin, float wmax) {
  float O = wmax - wmin, o = w - wmin;
  if (!(O > 0.f) || !(o > 0.f)) return 0u;
  int k = (int)(0.5f * log2f(O / o));
  return (uint32_t)max(0, 7 - k);
}

__global__ void pack_keys_kernel(const float* __restrict__ xyz, const float* __restrict__ w, int n,
                                 const SetInfo* __restrict__ sets, int nsets, int set_shift, int bin_shift,
                                 const unsigned* __restrict__ wr, uint64_t* __restrict__ keys, int* __restrict__ vals,
                                 unsigned* __restrict__ hist, int* __restrict__ counts, int* __restrict__ ovf_slot,
                                 DevStatus* st) {
  __shared__ unsigned h[8][256];  // the sort's digit counts
  for (int k = threadIdx.x; k < 8 * 256; k += blockDim.x) (&h[0][0])[k] = 0;
  __syncthreads();
  const int bits = bin_shift / 3;
  const float scale = (float)(1u << bits);
  const unsigned least = ~wr[0], most = wr[1];
  const float wmin = o2f(least), wmax = o2f(most);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    float x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
    int s = nsets > 1 ? find_set(sets, nsets, i) : 0;
    const SetInfo& S = sets[s];
    bool ok = isfinite(x) && isfinite(y) && isfinite(z);
    if (w && S.weighted) ok = ok && isfinite(w[i]);
    if (!ok) set_error(st, VD_ERR_INVALID_ARG);
    float c[3] = {x, y, z};
    uint32_t q[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
      float t = (c[k] - S.lo[k]) / (S.hi[k] - S.lo[k]);
      t = fminf(fmaxf(t, 0.0f), 1.0f);  // NaN -> 0 via fmaxf
      float v = floorf(t * scale);
      q[k] = (uint32_t)fminf(v, scale - 1.0f);
    }
    uint64_t code = (spread3(q[0]) << 2) | (spread3(q[1]) << 1) | spread3(q[2]);
    uint32_t bin = (w && S.weighted && least <= most) ? weight_bin(w[i], wmin, wmax) : 0u;
    const uint64_t key = ((uint64_t)s << set_shift) | ((uint64_t)bin << bin_shift) | code;
    keys[i] = key;
    vals[i] = i;
    counts[i] = 0;  // no neighbours, no place in the pool yet
    ovf_slot[i] = -1;
#pragma unroll
    for (int d = 0; d < 8; d++) atomicAdd(&h[d][(unsigned)(key >> (8 * d)) & 255u], 1u);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 8 * 256; k += blockDim.x) {
    const unsigned c = (&h[0][0])[k];
    if (c) atomicAdd(&hist[k], c);
  }
}

cudaError_t launch_pack_keys(const float* xyz, const float* w, int n, const SetInfo* sets, int nsets, int set_shift,
                             int bin_shift, const unsigned* wr, uint64_t* keys, int* vals, unsigned* hist, int* counts,
                             int* ovf_slot, DevStatus* st, cudaStream_t s) {
  int threads = 256;
  int blocks = min((n + threads - 1) / threads, 1024);
  pack_keys_kernel<<<blocks, threads, 0, s>>>(xyz, w, n, sets, nsets, set_shift, bin_shift, wr, keys, vals, hist,
                                              counts, ovf_slot, st);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- radix sort
//
// Stable LSD radix sort of (uint64 key, int value) pairs, 8-bit digits. The
// counts of all eight digits are taken while the keys are made
// (pack_keys_kernel), so that each digit is one pass over the array: a tile
// of keys is ranked by warp (__match_any_sync), the tiles' counts are chained
// by a look-back (each tile publishes its own counts, then the counts up to
// and including itself, and adds up what its predecessors have published),
// and the tile leaves in digit order, through shared memory. It is bound by
// the passes' reads and writes (24 bytes a site and pass) on large inputs
// and by launches on small ones. Measured against a pass in three kernels (count,
// a scan in one block, scatter by warps of 2,048 keys each; 24 launches): 10,000
// sites 390 -> 64 us, 1M 1.21 -> 0.19 ms, 20M 9.4 -> 2.2 ms (three times the
// time of the passes' bytes at the copy rate).
//
// Tiles are numbered in the order in which their blocks start, so a tile only
// waits for tiles that are running or done; the wait is bounded all the same.
// A tile whose wait runs out writes nothing: it reports VD_ERR_TIMEOUT and sets
// sort_failed, at which every later tile and pass stops (the arrays hold no
// permutation any more) and gather_sites_kernel starts from the input's order.

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr unsigned kSortOwn = 1u << 30, kSortSum = 2u << 30, kSortValue = (1u << 30) - 1u;
constexpr int kSortWaitLimit = 1 << 22;

template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) sort_pass_kernel(const uint64_t* __restrict__ keys,
                                                                 const int* __restrict__ vals, int n, int shift,
                                                                 const unsigned* __restrict__ hist,
                                                                 unsigned* __restrict__ ticket,
                                                                 volatile unsigned* __restrict__ chain,
                                                                 unsigned* __restrict__ next_chain,
                                                                 uint64_t* __restrict__ keys_out,
                                                                 int* __restrict__ vals_out, DevStatus* st) {
  constexpr int TILE = kSortThreads * ITEMS;
  __shared__ unsigned wh[kSortWarps][256];  // counts by warp, then each warp's first place in the tile
  __shared__ unsigned part[kSortWarps];
  __shared__ int place[256];  // where a digit's keys go, less their first place in the tile
  __shared__ uint64_t sk[TILE];
  __shared__ int sv[TILE];
  __shared__ int tile_id;
  const int t = (int)threadIdx.x, lane = t & 31, w = t >> 5;
  if (t == 0) {
    const int failed = *(volatile const int*)&st->sort_failed;
    const int id = (int)atomicAdd(ticket, 1u);
    tile_id = failed ? -1 : id;
  }
  for (int k = t; k < kSortWarps * 256; k += kSortThreads) (&wh[0][0])[k] = 0;
  __syncthreads();
  const int tile = tile_id;
  if (tile < 0) return;
  next_chain[(size_t)tile * 256 + t] = 0;  // the next pass's chain, idle during this one
  const int base = tile * TILE + w * 32 * ITEMS + lane;
  uint64_t key[ITEMS];
  int rank[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    const int at = base + 32 * i;
    key[i] = at < n ? keys[at] : ~0ull;
  }
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    const bool in = base + 32 * i < n;
    const unsigned d = in ? (unsigned)(key[i] >> shift) & 255u : 256u;
    const unsigned peers = __match_any_sync(FULL, d);
    const unsigned before = in ? wh[w][d] : 0u;
    rank[i] = (int)before + __popc(peers & lanemask_lt());
    __syncwarp();
    if (in && (peers >> lane) == 1u) wh[w][d] = before + __popc(peers);  // the highest peer
    __syncwarp();
  }
  __syncthreads();
  // thread t: digit t. Its places in the tile by warp, and its count
  unsigned count = 0;
#pragma unroll
  for (int q = 0; q < kSortWarps; q++) {
    const unsigned c = wh[q][t];
    wh[q][t] = count;
    count += c;
  }
  chain[(size_t)tile * 256 + t] = count | (tile == 0 ? kSortSum : kSortOwn);
  // exclusive sums over the digits, of the tile's counts and of all keys'
  const unsigned total = hist[t];
  unsigned a = count, b = total;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned x = __shfl_up_sync(FULL, a, o), y = __shfl_up_sync(FULL, b, o);
    if (lane >= o) {
      a += x;
      b += y;
    }
  }
  __shared__ unsigned part2[kSortWarps];
  if (lane == 31) {
    part[w] = a;
    part2[w] = b;
  }
  __syncthreads();
  a -= count;
  b -= total;
  for (int q = 0; q < w; q++) {
    a += part[q];
    b += part2[q];
  }
#pragma unroll
  for (int q = 0; q < kSortWarps; q++) wh[q][t] += a;
  unsigned sum = 0;
  bool lost = false;
  if (tile > 0) {
    int waits = 0;
    for (int p = tile - 1; p >= 0;) {
      const unsigned v = chain[(size_t)p * 256 + t];
      if (v < kSortOwn) {
        // a tile that stopped publishes nothing: look for the mark now and then
        if (++waits > kSortWaitLimit || ((waits & 1023) == 0 && *(volatile const int*)&st->sort_failed)) {
          lost = true;
          break;
        }
        continue;
      }
      sum += v & kSortValue;
      if (v >= kSortSum) break;
      p--;
    }
    if (!lost) chain[(size_t)tile * 256 + t] = (count + sum) | kSortSum;
  }
  place[t] = (int)(b + sum) - (int)a;
  if (__syncthreads_or(lost)) {
    if (t == 0) {
      set_error(st, VD_ERR_TIMEOUT);
      atomicExch(&st->sort_failed, 1);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    const int at = base + 32 * i;
    if (at < n) {
      const int to = rank[i] + (int)wh[w][(unsigned)(key[i] >> shift) & 255u];
      sk[to] = key[i];
      sv[to] = vals[at];
    }
  }
  __syncthreads();
  const int cnt = min(TILE, n - tile * TILE);
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    const int at = t + kSortThreads * i;
    if (at < cnt) {
      const uint64_t k = sk[at];
      const int to = min(max(at + place[(unsigned)(k >> shift) & 255u], 0), n - 1);
      keys_out[to] = k;
      vals_out[to] = sv[at];
    }
  }
}

// Tiles of 1,024 keys below 2^18 (more blocks at work), of 3,072 from there on
// (fewer links in the chain, whole sectors per digit): around 2^18 they take
// 0.12 and 0.13 ms.
static int sort_items(int n) { return n < (1 << 18) ? 4 : 12; }
static int sort_tiles(int n) { return (n + kSortThreads * sort_items(n) - 1) / (kSortThreads * sort_items(n)); }

size_t sort_scratch_bytes(int64_t n) {
  // histograms and tickets, then two chains
  const int64_t tiles = std::max<int64_t>(n / (kSortThreads * 12) + 1, std::min<int64_t>(n / (kSortThreads * 4) + 1, 257));
  return sizeof(unsigned) * (kSortHist + 2 * 256 * (size_t)tiles);
}

// Words at the head of the scratch that must start at 0: the digit counts that
// the keys' kernel adds to, the tickets and the first chain.
size_t sort_clear_words(int n) { return kSortHist + 256 * (size_t)sort_tiles(n); }

// All digits of at most kSortSmall keys in one block: 500 keys 29 -> 14 us (and
// seven launches less).
constexpr int kSortSmall = 2048;
__global__ void __launch_bounds__(512) sort_small_kernel(uint64_t* __restrict__ keys, int* __restrict__ vals, int n,
                                                         int bits) {
  constexpr int ITEMS = kSortSmall / 512, W = 16;
  __shared__ unsigned wh[W][256];
  __shared__ unsigned part[8];
  __shared__ uint64_t sk[kSortSmall];
  __shared__ int sv[kSortSmall];
  const int t = (int)threadIdx.x, lane = t & 31, w = t >> 5;
  const int base = w * 32 * ITEMS + lane;
  uint64_t key[ITEMS];
  int val[ITEMS], rank[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    const int at = base + 32 * i;
    key[i] = at < n ? keys[at] : ~0ull;
    val[i] = at < n ? vals[at] : 0;
  }
  for (int shift = 0; shift < bits; shift += 8) {
    for (int k = t; k < W * 256; k += 512) (&wh[0][0])[k] = 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      const bool in = base + 32 * i < n;
      const unsigned d = in ? (unsigned)(key[i] >> shift) & 255u : 256u;
      const unsigned peers = __match_any_sync(FULL, d);
      const unsigned before = in ? wh[w][d] : 0u;
      rank[i] = (int)before + __popc(peers & lanemask_lt());
      __syncwarp();
      if (in && (peers >> lane) == 1u) wh[w][d] = before + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    unsigned count = 0, a = 0;
    if (t < 256) {
#pragma unroll
      for (int q = 0; q < W; q++) {
        const unsigned c = wh[q][t];
        wh[q][t] = count;
        count += c;
      }
      a = count;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned x = __shfl_up_sync(FULL, a, o);
        if (lane >= o) a += x;
      }
      if (lane == 31) part[w] = a;
    }
    __syncthreads();
    if (t < 256) {
      a -= count;
      for (int q = 0; q < w; q++) a += part[q];
#pragma unroll
      for (int q = 0; q < W; q++) wh[q][t] += a;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; i++)
      if (base + 32 * i < n) {
        const int to = rank[i] + (int)wh[w][(unsigned)(key[i] >> shift) & 255u];
        sk[to] = key[i];
        sv[to] = val[i];
      }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      const int at = base + 32 * i;
      if (at < n) {
        key[i] = sk[at];
        val[i] = sv[at];
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    const int at = base + 32 * i;
    if (at < n) {
      keys[at] = key[i];
      vals[at] = val[i];
    }
  }
}

int sort_launches(int n, int bits) { return n <= 1 ? 0 : (n <= kSortSmall ? 1 : (bits + 7) / 8); }

cudaError_t radix_sort_pairs(uint64_t*& keys, uint64_t*& keys_alt, int*& vals, int*& vals_alt, unsigned* scratch, int n,
                             int bits, DevStatus* st, cudaStream_t s) {
  if (n <= 1) return cudaSuccess;
  if (n <= kSortSmall) {
    sort_small_kernel<<<1, 512, 0, s>>>(keys, vals, n, bits);
    return cudaGetLastError();
  }
  const int tiles = sort_tiles(n);
  unsigned* chain = scratch + kSortHist;
  unsigned* other = chain + 256 * (size_t)tiles;
  for (int shift = 0, d = 0; shift < bits; shift += 8, d++) {
    if (sort_items(n) == 4)
      sort_pass_kernel<4><<<tiles, kSortThreads, 0, s>>>(keys, vals, n, shift, scratch + 256 * d, scratch + 2048 + d, chain,
                                                        other, keys_alt, vals_alt, st);
    else
      sort_pass_kernel<12><<<tiles, kSortThreads, 0, s>>>(keys, vals, n, shift, scratch + 256 * d, scratch + 2048 + d, chain,
                                                         other, keys_alt, vals_alt, st);
    std::swap(keys, keys_alt);
    std::swap(vals, vals_alt);
    std::swap(chain, other);
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------- packed sorted sites
//
// The packed site of every sorted place, the inverse permutation, and the
// losers of duplicate positions: sites at exactly the same position (and
// weight stratum) share a key and are adjacent after the sort. Among them the
// larger weight, then the lower original index, keeps its cell; every other
// one has an empty cell, and its half-space is implied by the winner's, so it
// is never a candidate.
//
// After a sort that gave up (`failed`), perm and keys hold whatever was in the
// arrays: every place takes the input's own order instead, with keys of the
// set alone (sorted, so the tree over them is a valid one), and every site is a
// loser, so that no cell is made of it: the build ends with empty rows and
// VD_ERR_TIMEOUT. (This function makes place k. It is compiled for the host too,
// where a test runs it on such arrays.)
__host__ __device__ inline void gather_site(const float* xyz, const float* w, int* perm, int n, const SetInfo* sets,
                                            uint64_t* keys, int set_shift, int nsets, bool failed, float4* sites,
                                            int* inv, unsigned char* loser, int k) {
  if (failed) {
    perm[k] = k;
    keys[k] = nsets > 1 ? (uint64_t)find_set(sets, nsets, k) << set_shift : 0;
  }
  const int i = perm[k];
  const uint64_t key = keys[k];
  const int s = nsets > 1 ? (int)(key >> set_shift) : 0;
  const bool weighted = w && sets[s].weighted;
  const float4 p = make_float4(xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], weighted ? w[i] : 0.0f);
  sites[k] = p;
  inv[i] = k;
  bool lose = failed;
  for (int dir = -1; dir <= 1 && !lose; dir += 2)
    for (int m = k + dir; m >= 0 && m < n && keys[m] == key && !lose; m += dir) {
      const int o = perm[m];
      if (xyz[3 * o] == p.x && xyz[3 * o + 1] == p.y && xyz[3 * o + 2] == p.z) {
        const float qw = weighted ? w[o] : 0.0f;
        lose = qw > p.w || (qw == p.w && o < i);
      }
    }
  loser[k] = lose ? 1 : 0;
}

__global__ void gather_sites_kernel(const float* __restrict__ xyz, const float* __restrict__ w, int* __restrict__ perm,
                                    int n, const SetInfo* __restrict__ sets, uint64_t* __restrict__ keys, int set_shift,
                                    int nsets, const DevStatus* __restrict__ st, float4* __restrict__ sites,
                                    int* __restrict__ inv, unsigned char* __restrict__ loser) {
  const bool failed = st->sort_failed != 0;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
    gather_site(xyz, w, perm, n, sets, keys, set_shift, nsets, failed, sites, inv, loser, k);
}

cudaError_t launch_gather_sites(const float* xyz, const float* w, int* perm, int n, const SetInfo* sets, uint64_t* keys,
                                int set_shift, int nsets, const DevStatus* st, float4* sites, int* inv,
                                unsigned char* loser, cudaStream_t s) {
  int threads = 256;
  int blocks = min((n + threads - 1) / threads, 4096);
  gather_sites_kernel<<<blocks, threads, 0, s>>>(xyz, w, perm, n, sets, keys, set_shift, nsets, st, sites, inv, loser);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- Karras radix tree

__device__ __forceinline__ int common_prefix(const uint64_t* keys, int n, int i, int j) {
  if (j < 0 || j >= n) return -1;
  uint64_t a = keys[i], b = keys[j];
  if (a != b) return __clzll((long long)(a ^ b));
  return 64 + __clz(i ^ j);
}

// Internal node i of the binary radix tree over n sorted keys (ties broken
// by position). Children: internal index >= 0, or -1-site for a single site.
__global__ void karras_kernel(const uint64_t* __restrict__ keys, int n, int* __restrict__ left,
                              int* __restrict__ right, int* __restrict__ parent, int2* __restrict__ range,
                              int* __restrict__ visit) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n - 1) return;
  visit[i] = 0;
  int dplus = common_prefix(keys, n, i, i + 1), dminus = common_prefix(keys, n, i, i - 1);
  int d = dplus > dminus ? 1 : -1;
  int dmin = min(dplus, dminus);
  int lmax = 2;
  while (common_prefix(keys, n, i, i + lmax * d) > dmin) lmax <<= 1;
  int l = 0;
  for (int t = lmax >> 1; t >= 1; t >>= 1)
    if (common_prefix(keys, n, i, i + (l + t) * d) > dmin) l += t;
  int j = i + l * d;
  int dnode = common_prefix(keys, n, i, j);
  int s = 0;
  int t = l;
  do {
    t = (t + 1) >> 1;
    if (common_prefix(keys, n, i, i + (s + t) * d) > dnode) s += t;
  } while (t > 1);
  int gamma = i + s * d + min(d, 0);
  int lo = min(i, j), hi = max(i, j);
  int lc = (lo == gamma) ? (-1 - gamma) : gamma;
  int rc = (hi == gamma + 1) ? (-1 - (gamma + 1)) : (gamma + 1);
  left[i] = lc;
  right[i] = rc;
  range[i] = make_int2(lo, hi);
  // parent array: internal nodes at [0, n-1), sites at [n-1, 2n-1)
  parent[lc >= 0 ? lc : (n - 1) + (-1 - lc)] = i;
  parent[rc >= 0 ? rc : (n - 1) + (-1 - rc)] = i;
  if (i == 0) parent[0] = -1;
}

__device__ __forceinline__ void child_box(int c, const float4* sites, const float4* box_lo, const float4* box_hi,
                                          float4& lo, float4& hi) {
  if (c < 0) {
    float4 p = sites[-1 - c];
    lo = p;
    hi = make_float4(p.x, p.y, p.z, 0.0f);
  } else {
    lo = __ldcg(&box_lo[c]);
    hi = __ldcg(&box_hi[c]);
  }
}

// Bottom-up AABB + max-weight refit: the second visitor of a node merges
// its two children and walks on (no spinning on other threads).
__global__ void refit_kernel(const float4* __restrict__ sites, const int* __restrict__ left,
                             const int* __restrict__ right, const int* __restrict__ parent, int* visit,
                             float4* box_lo, float4* box_hi, int n) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  int p = parent[(n - 1) + k];
  while (p >= 0) {
    __threadfence();
    if (atomicAdd(&visit[p], 1) == 0) return;
    __threadfence();
    float4 a0, a1, b0, b1;
    child_box(left[p], sites, box_lo, box_hi, a0, a1);
    child_box(right[p], sites, box_lo, box_hi, b0, b1);
    float4 lo = make_float4(fminf(a0.x, b0.x), fminf(a0.y, b0.y), fminf(a0.z, b0.z), fmaxf(a0.w, b0.w));
    float4 hi = make_float4(fmaxf(a1.x, b1.x), fmaxf(a1.y, b1.y), fmaxf(a1.z, b1.z), 0.0f);
    __stcg(&box_lo[p], lo);
    __stcg(&box_hi[p], hi);
    p = parent[p];
  }
}

// 8-wide traversal record of internal node i: the nodes three binary levels
// below it, or the leaf (at most kWideLeaf sites) a path ends at earlier, in
// the slot of that path followed by zeros; the other slots are empty. Eight
// boxes' low corners (w: maximum weight), then their high corners (w:
// reference), so that eight lanes read each half as one 128-byte line.
// The binary record (both children's boxes, max weights and references: 64
// bytes, read by four lanes with one float4 each) by the first two of the
// eight threads.
__device__ __forceinline__ void emit_node(int i, int s, const float4* __restrict__ sites, const int* __restrict__ left,
                                          const int* __restrict__ right, const int2* __restrict__ range,
                                          const float4* __restrict__ box_lo, const float4* __restrict__ box_hi,
                                          int leaf_size, float4* __restrict__ nodes, float4* __restrict__ wide) {
  if (s < 2) {
    const int ch = s == 0 ? left[i] : right[i];
    float4 lo, hi;
    int ref;
    if (ch < 0) {
      lo = sites[-1 - ch];
      hi = lo;
      ref = make_leaf_ref(-1 - ch, 1);
    } else {
      lo = box_lo[ch];
      hi = box_hi[ch];
      const int2 r = range[ch];
      const int cnt = r.y - r.x + 1;
      ref = cnt <= leaf_size ? make_leaf_ref(r.x, cnt) : ch;
    }
    hi.w = __int_as_float(ref);
    nodes[4 * (size_t)i + 2 * s] = lo;
    nodes[4 * (size_t)i + 2 * s + 1] = hi;
  }
  const int2 own = range[i];
  if (!wide || own.y - own.x < kWideLeaf) return;  // inside a leaf: never visited
  int c = i, first = own.x, cnt = own.y - own.x + 1;
  bool valid = true;
#pragma unroll
  for (int b = 2; b >= 0; b--) {
    if (cnt <= kWideLeaf) {
      valid = valid && ((s >> b) & 1) == 0;
      continue;
    }
    c = (s >> b) & 1 ? right[c] : left[c];
    if (c < 0) {
      first = -1 - c;
      cnt = 1;
    } else {
      const int2 r = range[c];
      first = r.x;
      cnt = r.y - r.x + 1;
    }
  }
  float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
  int ref = kNoChild;
  if (valid) {
    if (c < 0) {
      lo = sites[first];
      hi = lo;
    } else {
      lo = box_lo[c];
      hi = box_hi[c];
    }
    ref = cnt <= kWideLeaf ? make_leaf_ref(first, cnt) : c;
  }
  hi.w = __int_as_float(ref);
  wide[16 * (size_t)i + s] = lo;
  wide[16 * (size_t)i + 8 + s] = hi;
}

// Root references of every set: the node whose range is exactly the set.
__device__ __forceinline__ void set_root(SetInfo* sets, int s, const int2* __restrict__ range, int n, int leaf_size,
                                         DevStatus* st) {
  int f = sets[s].first, c = sets[s].count;
  if (c <= 0) {
    sets[s].root = sets[s].wroot = 0;
    return;
  }
  int l = f + c - 1, node = -1;
  if (f < n - 1) {
    const int2 r = range[f];
    if (r.x == f && r.y == l) node = f;
  }
  if (node < 0 && l < n - 1) {
    const int2 r = range[l];
    if (r.x == f && r.y == l) node = l;
  }
  if (node < 0 && c > min(leaf_size, kWideLeaf)) {
    node = 0;
    set_error(st, VD_ERR_INVALID_ARG);
  }
  sets[s].root = c <= leaf_size ? make_leaf_ref(f, c) : node;
  sets[s].wroot = c <= kWideLeaf ? make_leaf_ref(f, c) : node;
}

// The same boxes for small inputs, without the climb's chain of fences and
// round trips (500 sites 22 us, 10,000 32 us): each node reads all of its sites.
__global__ void __launch_bounds__(128) node_boxes_kernel(const float4* __restrict__ sites, const int2* __restrict__ range,
                                                         float4* __restrict__ box_lo, float4* __restrict__ box_hi) {
  __shared__ float part[7][4];
  const int2 r = range[blockIdx.x];
  const int t = (int)threadIdx.x;
  float v[7];  // low corner, negated high corner, negated weight
#pragma unroll
  for (int k = 0; k < 7; k++) v[k] = INFINITY;
#pragma unroll 4
  for (int j = r.x + t; j <= r.y; j += 128) {
    const float4 p = sites[j];
    v[0] = fminf(v[0], p.x);
    v[1] = fminf(v[1], p.y);
    v[2] = fminf(v[2], p.z);
    v[3] = fminf(v[3], -p.x);
    v[4] = fminf(v[4], -p.y);
    v[5] = fminf(v[5], -p.z);
    v[6] = fminf(v[6], -p.w);
  }
#pragma unroll
  for (int k = 0; k < 7; k++) {
    for (int o = 16; o > 0; o >>= 1) v[k] = fminf(v[k], __shfl_xor_sync(FULL, v[k], o));
    if ((t & 31) == 0) part[k][t >> 5] = v[k];
  }
  __syncthreads();
  if (t == 0) {
#pragma unroll
    for (int k = 0; k < 7; k++) v[k] = fminf(fminf(part[k][0], part[k][1]), fminf(part[k][2], part[k][3]));
    box_lo[blockIdx.x] = make_float4(v[0], v[1], v[2], -v[6]);
    box_hi[blockIdx.x] = make_float4(-v[3], -v[4], -v[5], 0.0f);
  }
}
constexpr int kBoxesDirect = 16384;  // where they take 13 and 34 us; a node's work grows with its sites

// The traversal records, and the sets' roots.
__global__ void emit_kernel(const float4* __restrict__ sites, const int* __restrict__ left,
                            const int* __restrict__ right, const int2* __restrict__ range,
                            const float4* __restrict__ box_lo, const float4* __restrict__ box_hi, int n, int leaf_size,
                            float4* __restrict__ nodes, float4* __restrict__ wide, SetInfo* sets, int nsets,
                            DevStatus* st) {
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid < nsets) set_root(sets, (int)tid, range, n, leaf_size, st);
  const int i = (int)(tid >> 3);
  if (i < n - 1) emit_node(i, (int)(tid & 7), sites, left, right, range, box_lo, box_hi, leaf_size, nodes, wide);
}

cudaError_t launch_build_bvh(const uint64_t* keys, const float4* sites, int n, int leaf_size, BvhBuffers& b,
                             SetInfo* sets, int nsets, DevStatus* st, cudaStream_t s) {
  int threads = 256;
  if (n >= 2) {
    int blocks = (n - 1 + threads - 1) / threads;
    karras_kernel<<<blocks, threads, 0, s>>>(keys, n, b.left, b.right, b.parent, b.range, b.visit);
    if (n <= kBoxesDirect)
      node_boxes_kernel<<<n - 1, 128, 0, s>>>(sites, b.range, b.box_lo, b.box_hi);
    else
      refit_kernel<<<(n + threads - 1) / threads, threads, 0, s>>>(sites, b.left, b.right, b.parent, b.visit,
                                                                    b.box_lo, b.box_hi, n);
  }
  const long long work = std::max<long long>(8ll * (n - 1), nsets);
  emit_kernel<<<(int)((work + threads - 1) / threads), threads, 0, s>>>(sites, b.left, b.right, b.range, b.box_lo, b.box_hi,
                                                                       n, leaf_size, b.nodes, b.wide, sets, nsets, st);
  return cudaGetLastError();
}

}  // namespace vd
