// vd_noalloc.cu -- vd_cells_noalloc: cells of a small point set without any
// device allocation.
//
// Some callers cannot call cudaMalloc: code running inside another
// framework's memory pool or allocator hooks, real-time or safety-critical
// loops that forbid allocation after start-up, and callers that must not
// create a context workspace at all. For them this entry point keeps all of
// its scratch (the packed sites, a duplicate mask, a work counter and a
// status block) in one file-scope device array of fixed size, and writes
// only into the buffers the caller passes.
//
// The cells are made by the one-cell-per-warp kernel (vd_solo.cu) in its form
// without a tree, in which every other site is read (no sort or tree buffers
// are needed): 4,001 sites 1,120 -> 195 us, against a kernel of its own that
// clipped by the sites in index order. Cells that outgrow its capacity, or have more than
// VD_NOALLOC_ROW neighbours, are reported in the status word instead of moving
// to the large-cell path (which needs an arena).
#include <cuda.h>  // CUcontext / CUresult types of the two driver calls looked up below

#include <cstddef>
#include <cstring>
#include <mutex>

#include "vd_internal.cuh"

namespace vd {
namespace {

constexpr int kNaMaxSites = VD_NOALLOC_MAX_SITES;
constexpr int kNaRow = VD_NOALLOC_ROW;

struct NoAllocScratch {
  float4 sites[kNaMaxSites];         // packed (x, y, z, w), by site index
  SetInfo set;                       // the one set: its box and sites
  unsigned char loser[kNaMaxSites];  // an exact duplicate site beats this one
  int work;                          // persistent-grid work counter
  DevStatus st;                      // first device-side error (and counts)
};

// The scratch array itself. In host code `g_scratch` names a host-side
// stand-in, not device memory: the device address comes from
// cudaGetSymbolAddress (see scratch_on_device below).
static __device__ __align__(256) unsigned char g_scratch[sizeof(NoAllocScratch)];

// Pack the sites and find the losers of duplicate positions (the larger
// weight, then the lower index, keeps the cell): a warp per site, the others
// one per lane (a thread per site reading all others took 60% of a call).
__global__ void na_pack_kernel(const float* __restrict__ xyz, const float* __restrict__ w, int n, vd_box box,
                               NoAllocScratch* S) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    for (int k = 0; k < 3; k++) {
      S->set.lo[k] = box.lo[k];
      S->set.hi[k] = box.hi[k];
    }
    S->set.first = 0;
    S->set.count = n;
    S->set.root = S->set.wroot = 0;
    S->set.weighted = w ? 1 : 0;
  }
  const int lane = (int)lane_id();
  for (int i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); i < n; i += (int)((gridDim.x * blockDim.x) >> 5)) {
    const float x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
    const float wi = w ? w[i] : 0.0f;
    bool lose = false;
#pragma unroll 4
    for (int j = lane; j < n; j += 32)
      if (xyz[3 * j] == x && xyz[3 * j + 1] == y && xyz[3 * j + 2] == z && j != i) {
        const float wj = w ? w[j] : 0.0f;
        lose = lose || wj > wi || (wj == wi && j < i);
      }
    lose = __any_sync(FULL, lose);
    if (lane == 0) {
      if (!(isfinite(x) && isfinite(y) && isfinite(z) && isfinite(wi))) set_error(&S->st, VD_ERR_INVALID_ARG);
      S->sites[i] = make_float4(x, y, z, wi);
      S->loser[i] = lose ? 1 : 0;
    }
  }
}

__global__ void na_status_kernel(const NoAllocScratch* S, int32_t* status) { *status = S->st.error; }

// Device address of the scratch array on the current device. It is looked
// up once per device and CUDA context (with that device current) and cached;
// a cudaDeviceReset gives the device a new context (and the module a new
// copy of the array), so the cache is keyed by the context's id, read through
// two driver calls that the runtime hands out (no link to the driver
// library). If that id cannot be read, the address is looked up on every
// call, which allocates nothing either.
typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);

std::mutex g_mu;
struct ScratchSlot {
  void* addr;
  unsigned long long ctx_id;
};
ScratchSlot g_slot[64] = {};
CtxGetCurrentFn g_get_current = nullptr;
CtxGetIdFn g_get_id = nullptr;
bool g_entry_tried = false;

bool context_id(unsigned long long* id) {
  if (!g_entry_tried) {
    g_entry_tried = true;
    cudaDriverEntryPointQueryResult q;
    void* f = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      g_get_current = reinterpret_cast<CtxGetCurrentFn>(f);
    f = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      g_get_id = reinterpret_cast<CtxGetIdFn>(f);
  }
  CUcontext c = nullptr;
  if (!g_get_current || !g_get_id || g_get_current(&c) != CUDA_SUCCESS || !c) return false;
  return g_get_id(c, id) == CUDA_SUCCESS;
}

int scratch_on_device(NoAllocScratch** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return VD_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_mu);
  unsigned long long id = 0;
  const bool have_id = context_id(&id);
  ScratchSlot& S = g_slot[dev];
  if (!S.addr || !have_id || S.ctx_id != id) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_scratch) != cudaSuccess || !p) return VD_ERR_CUDA;
    S.addr = p;
    S.ctx_id = have_id ? id : 0;
  }
  *out = static_cast<NoAllocScratch*>(S.addr);
  return VD_OK;
}

}  // namespace
}  // namespace vd

using namespace vd;

extern "C" int vd_cells_noalloc(const float* sites_xyz, const float* weights, int64_t n, vd_box bbox,
                                int32_t* counts, int32_t* neighbors, float* volume, float* centroid,
                                int32_t* status, void* stream) {
  if (!sites_xyz || !counts || !neighbors || !volume || !centroid || !status || n <= 0) return VD_ERR_INVALID_ARG;
  if (n > kNaMaxSites) return VD_ERR_TOO_LARGE;
  for (int k = 0; k < 3; k++)
    if (!(bbox.lo[k] < bbox.hi[k])) return VD_ERR_INVALID_ARG;
  NoAllocScratch* S = nullptr;
  int rc = scratch_on_device(&S);
  if (rc) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // the work counter and the status block must start at zero on every call
  if (cudaMemsetAsync(&S->work, 0, sizeof(NoAllocScratch) - offsetof(NoAllocScratch, work), s) != cudaSuccess)
    return VD_ERR_CUDA;
  int nn = (int)n;
  int sms = 0, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                 cudaSuccess)
    return VD_ERR_CUDA;
  // each launch through cudaLaunchKernel, whose return value is that
  // launch's own status: an error left by the caller's earlier work is
  // neither reported as ours nor cleared
  const float* w = weights;
  void* pack_args[] = {(void*)&sites_xyz, (void*)&w, (void*)&nn, (void*)&bbox, (void*)&S};
  if (cudaLaunchKernel((const void*)na_pack_kernel, dim3((nn + 7) / 8), dim3(256), pack_args, 0, s) !=
      cudaSuccess)
    return VD_ERR_CUDA;
  CellBuffers c;
  std::memset(&c, 0, sizeof(c));
  c.sites = S->sites;
  c.loser = S->loser;
  c.sets = &S->set;
  c.nsets = 1;
  c.n = nn;
  c.counts = counts;
  c.scratch = neighbors;
  c.stride = kNaRow;
  c.vol = volume;
  c.cen = centroid;
  c.work = &S->work;
  c.st = &S->st;
  c.cell_end = nn;
  if (launch_solo_brute(c, sms, s) != cudaSuccess) return VD_ERR_CUDA;
  const NoAllocScratch* Sc = S;
  void* st_args[] = {(void*)&Sc, (void*)&status};
  if (cudaLaunchKernel((const void*)na_status_kernel, dim3(1), dim3(1), st_args, 0, s) != cudaSuccess)
    return VD_ERR_CUDA;
  return VD_OK;
}
