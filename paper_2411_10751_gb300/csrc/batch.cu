// Batched step: many independent periodic D2Q37 domains (any sizes, sources
// and parameters) advanced by ONE persistent launch per time step, replayed
// from a CUDA graph.  Resident CTAs (all of the same shape: 352 threads) take
// (domain, tile) items from a global work list in order through a device
// counter and run the step without staging (direct_tile, step2d_direct.cuh) of
// the domain's source kind on it: most tiles of small domains touch the
// periodic edge or belong to rows that TMA cannot take, so staging them was a
// synchronous gather into shared memory, and a block held 93 KB of it.  A tile's
// 256 nodes take one thread each; the theta ring of the thermal kind runs
// beside them on the last three warps, the 276 psi nodes of the pseudopotential
// kind before them on all.  The pseudopotential tiles, the slowest, come first
// in the work list, so the launch ends on short tiles.  Item and step arguments
// are read from device memory one item ahead, by the last warps while the
// others collide.  It is bound by instruction issue (half of the slots) and the
// loads' latency at 22 warps per SM: 256 domains, 6.4 M nodes, FP32, 770 us a step
// staged, 564 us pulled, 522 us with 32-bit offsets in the pulls (FP16 484; three
// CTAs per SM at 56 registers 559 and 509).  Batches of large aligned domains gain
// less, since their tiles could be staged (us per step, staged / pulled, four
// domains of 1024 x 1024: thermal 325 / 273, body force 304 / 243, pseudopotential
// 379 / 383; of 512 x 512 90.6 / 72.6 thermal, 106 / 99.9 pseudopotential).
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "hlbm.h"
#include "internal.h"
#include "step2d_direct.cuh"

namespace hlbm {
namespace {

constexpr int kThreads = Direct2<KIND_THERMAL>::NT;
constexpr int kOwn = Direct2<KIND_THERMAL>::OWN;
constexpr int kAux = Direct2<KIND_SC>::Fr::SW * Direct2<KIND_SC>::Fr::SH;

struct BatchDomain {
  StepArgs args[2];       // args[0]: from the buffer that holds the state at the start of the batch call, args[1]: back
};
struct BatchItem {
  int domain, kind, x0, y0;
};
constexpr int kArgWords = (int)(sizeof(StepArgs) / 4);
static_assert(sizeof(StepArgs) % 8 == 0 && sizeof(BatchItem) == 16, "copied by words");

// One step of every domain: CTAs take work-list items (T = nitems) through
// the counter; a launch of G CTAs takes exactly T + G values (each CTA ends
// on one value past the list), so the counter is never reset and the item is
// the value modulo T + G.
template <int ST>
__global__ void __launch_bounds__(kThreads, 2)
    batch_step_kernel(const BatchDomain* __restrict__ doms, const BatchItem* __restrict__ items, int nitems, int flip,
                      unsigned long long* ctr) {
  __shared__ float aux[kAux];
  __shared__ __align__(16) unsigned s_args[2][kArgWords];
  __shared__ BatchItem s_item[2];
  __shared__ int s_next[4];                            // item index of turn n at n mod 4
  const int tid = threadIdx.x;
  // thread 0 takes item indices two turns ahead and keeps the last as the
  // counter's raw value, so the atomic's round trip overlaps a whole tile
  unsigned long long raw = 0;
  const unsigned long long period = (unsigned long long)nitems + gridDim.x;
  const auto fetch = [&](int turn, int first, int n) {   // threads first .. first + n - 1: item and arguments of a turn
    const int gi = s_next[turn & 3];
    if (gi >= nitems) return;
    const BatchItem it = items[gi];
    const unsigned* src = reinterpret_cast<const unsigned*>(&doms[it.domain].args[flip]);
    for (int w = tid - first; w < kArgWords; w += n) s_args[turn & 1][w] = __ldg(src + w);
    if (tid == first) s_item[turn & 1] = it;
  };
  if (tid == 0) {
    const int g0 = (int)(atomicAdd(ctr, 1ull) % period);
    s_next[0] = g0;
    if (g0 < nitems) raw = atomicAdd(ctr, 1ull);
  }
  __syncthreads();
  fetch(0, 0, kThreads);
  for (int turn = 0;; ++turn) {
    if (tid == 0 && s_next[turn & 3] < nitems) {
      const int gi = (int)(raw % period);
      s_next[(turn + 1) & 3] = gi;   // (a slow warp may still read the slot of turn - 1)
      if (gi < nitems) raw = atomicAdd(ctr, 1ull);
    }
    __syncthreads();   // this turn's item and the next one's index are there; aux is free
    if (s_next[turn & 3] >= nitems) return;
    const StepArgs& a = *reinterpret_cast<const StepArgs*>(s_args[turn & 1]);
    const BatchItem it = s_item[turn & 1];
    if (it.kind == KIND_SC) direct_tile<ST, KIND_SC, kThreads>(a, aux, it.x0, it.y0);
    else if (it.kind == KIND_THERMAL) direct_tile<ST, KIND_THERMAL, kThreads>(a, aux, it.x0, it.y0);
    else direct_tile<ST, KIND_LOCAL, kThreads>(a, aux, it.x0, it.y0);
    if (tid >= kOwn) fetch(turn + 1, kOwn, kThreads - kOwn);
  }
}

template <int ST>
int batch_grid(int nitems) {
  int per_sm = 0, sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_step_kernel<ST>, kThreads, 0);
  if (per_sm < 1) per_sm = 1;
  return std::max(1, std::min(nitems, sms * per_sm));
}

template <int ST>
cudaError_t launch_batch(const BatchDomain* doms, const BatchItem* items, int nitems, int grid, int flip,
                         unsigned long long* ctr, cudaStream_t s) {
  if (nitems <= 0) return cudaSuccess;
  batch_step_kernel<ST><<<grid, kThreads, 0, s>>>(doms, items, nitems, flip, ctr);
  return cudaGetLastError();
}

}  // namespace

// Host-side helpers the C ABI (api.cu) uses; the batch owns the device arrays.
struct BatchDevice {
  BatchDomain* doms = nullptr;
  BatchItem* items = nullptr;
  unsigned long long* ctr = nullptr;   // the persistent launch's item counter (zeroed once)
  int nitems = 0;
};

cudaError_t batch_upload(const std::vector<BatchDomain>& host, const std::vector<BatchItem>& items, BatchDevice& dev,
                         cudaStream_t s) {
  if (!dev.doms) {
    cudaError_t e = cudaMalloc(&dev.doms, host.size() * sizeof(BatchDomain));
    if (e != cudaSuccess) return e;
    e = cudaMalloc(&dev.items, items.size() * sizeof(BatchItem));
    if (e != cudaSuccess) return e;
    e = cudaMalloc(&dev.ctr, sizeof(unsigned long long));
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(dev.ctr, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = cudaMemcpyAsync(dev.doms, host.data(), host.size() * sizeof(BatchDomain), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(dev.items, items.data(), items.size() * sizeof(BatchItem), cudaMemcpyHostToDevice, s);
  dev.nitems = (int)items.size();
  return e;
}

}  // namespace hlbm

// ----------------------------------------------------------------- C ABI
using namespace hlbm;

struct hlbm_batch {
  std::vector<hlbm_ctx*> ctxs;
  int storage = 0;
  cudaStream_t stream = nullptr;
  std::vector<BatchDomain> host;
  std::vector<BatchItem> items;   // the pseudopotential kind's tiles first
  int grid = 0;                   // resident CTAs of the persistent launch
  BatchDevice dev;
  cudaGraphExec_t graph = nullptr;
  std::string msg;
};

// accessors of hlbm_ctx implemented in api.cu
namespace hlbm {
bool ctx_batchable(const hlbm_ctx* c, int* storage, int* kind, int* nx, int* ny);
StepArgs ctx_step_args(hlbm_ctx* c, int parity);
int ctx_cur(const hlbm_ctx* c);
void ctx_advance(hlbm_ctx* c, int steps);
}  // namespace hlbm

extern "C" {

hlbm_status hlbm_batch_create(int n, hlbm_ctx* const* ctxs, hlbm_batch** out) {
  if (!out || n < 1 || !ctxs) return HLBM_EINVAL;
  *out = nullptr;
  int storage = -1;
  for (int k = 0; k < n; ++k) {
    int st, kind, nx, ny;
    if (!ctxs[k] || !ctx_batchable(ctxs[k], &st, &kind, &nx, &ny)) {
      std::fprintf(stderr, "hlbm_batch_create: context %d is not an initialised periodic D2Q37 context\n", k);
      return HLBM_EINVAL;
    }
    if (storage >= 0 && st != storage) {
      std::fprintf(stderr, "hlbm_batch_create: all contexts must share one storage type\n");
      return HLBM_EINVAL;
    }
    storage = st;
  }
  hlbm_batch* b = new (std::nothrow) hlbm_batch();
  if (!b) return HLBM_ENOMEM;
  b->ctxs.assign(ctxs, ctxs + n);
  b->storage = storage;
  if (cudaStreamCreate(&b->stream) != cudaSuccess) {
    delete b;
    return HLBM_ECUDA;
  }
  for (hlbm_ctx* c : b->ctxs) {
    hlbm_synchronize(c);
    hlbm_set_stream(c, b->stream);
  }
  *out = b;
  return HLBM_OK;
}

static hlbm_status batch_refresh(hlbm_batch* b) {
  b->host.assign(b->ctxs.size(), BatchDomain{});
  b->items.clear();
  std::vector<BatchItem> heavy, light;   // pseudopotential tiles (the longest) and the others
  for (int kind : {(int)KIND_SC, (int)KIND_THERMAL, (int)KIND_LOCAL}) {
    for (size_t k = 0; k < b->ctxs.size(); ++k) {
      hlbm_ctx* c = b->ctxs[k];
      int st, dkind, nx, ny;
      ctx_batchable(c, &st, &dkind, &nx, &ny);
      if (dkind != kind) continue;
      BatchDomain& d = b->host[k];
      std::memset(&d, 0, sizeof(d));
      const int cur = ctx_cur(c);
      d.args[0] = ctx_step_args(c, cur);
      d.args[1] = ctx_step_args(c, cur ^ 1);
      for (int y0 = 0; y0 < ny; y0 += 8)
        for (int x0 = 0; x0 < nx; x0 += 32) (dkind == KIND_SC ? heavy : light).push_back(BatchItem{(int)k, dkind, x0, y0});
    }
  }
  // the slow tiles first, so the launch ends on short ones (against spreading them
  // evenly among the others, 256 domains, us per step: FP16 484 / 493, FP32 522 / 509)
  b->items = heavy;
  b->items.insert(b->items.end(), light.begin(), light.end());
  if (b->grid == 0)
    b->grid = b->storage == ST_F32 ? batch_grid<ST_F32>((int)b->items.size())
              : b->storage == ST_F16 ? batch_grid<ST_F16>((int)b->items.size())
                                     : batch_grid<ST_BF16>((int)b->items.size());
  cudaError_t e = batch_upload(b->host, b->items, b->dev, b->stream);
  if (e != cudaSuccess) {
    b->msg = std::string("batch upload: ") + cudaGetErrorString(e);
    return HLBM_ECUDA;
  }
  return HLBM_OK;
}

static cudaError_t batch_launch(hlbm_batch* b, int flip) {
  const int n = b->dev.nitems;
  switch (b->storage) {
    case ST_F32: return launch_batch<ST_F32>(b->dev.doms, b->dev.items, n, b->grid, flip, b->dev.ctr, b->stream);
    case ST_F16: return launch_batch<ST_F16>(b->dev.doms, b->dev.items, n, b->grid, flip, b->dev.ctr, b->stream);
    default: return launch_batch<ST_BF16>(b->dev.doms, b->dev.items, n, b->grid, flip, b->dev.ctr, b->stream);
  }
}

hlbm_status hlbm_batch_step(hlbm_batch* b, int n) {
  NvtxRange range("hlbm_batch_step");
  if (!b || n < 0) return HLBM_EINVAL;
  if (n == 0) return HLBM_OK;
  hlbm_status st = batch_refresh(b);
  if (st != HLBM_OK) return st;
  if (b->graph) {
    cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
  }
  // graph of two steps (buffer parity returns); odd remainder launched directly
  if (n >= 2) {
    if (cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return HLBM_ECUDA;
    cudaError_t le = batch_launch(b, 0);
    if (le == cudaSuccess) le = batch_launch(b, 1);
    cudaGraph_t g = nullptr;
    cudaError_t ce = cudaStreamEndCapture(b->stream, &g);
    if (le != cudaSuccess || ce != cudaSuccess) {
      b->msg = std::string("batch capture: ") + cudaGetErrorString(le != cudaSuccess ? le : ce);
      if (g) cudaGraphDestroy(g);
      return HLBM_ECUDA;
    }
    cudaError_t ie = cudaGraphInstantiate(&b->graph, g, 0);
    cudaGraphDestroy(g);
    if (ie != cudaSuccess) {
      b->graph = nullptr;
      return HLBM_ECUDA;
    }
    for (int k = 0; k < n / 2; ++k)
      if (cudaGraphLaunch(b->graph, b->stream) != cudaSuccess) return HLBM_ECUDA;
  }
  if (n % 2)
    if (batch_launch(b, 0) != cudaSuccess) return HLBM_ECUDA;
  for (hlbm_ctx* c : b->ctxs) ctx_advance(c, n);
  return HLBM_OK;
}

hlbm_status hlbm_batch_synchronize(hlbm_batch* b) {
  if (!b) return HLBM_EINVAL;
  if (cudaStreamSynchronize(b->stream) != cudaSuccess) return HLBM_ECUDA;
  for (hlbm_ctx* c : b->ctxs) {
    hlbm_status st = hlbm_synchronize(c);
    if (st != HLBM_OK) return st;
  }
  return HLBM_OK;
}

void* hlbm_batch_get_stream(hlbm_batch* b) { return b ? b->stream : nullptr; }

hlbm_status hlbm_batch_destroy(hlbm_batch* b) {
  if (!b) return HLBM_EINVAL;
  if (b->stream) cudaStreamSynchronize(b->stream);
  for (hlbm_ctx* c : b->ctxs) hlbm_set_stream(c, nullptr);
  if (b->graph) cudaGraphExecDestroy(b->graph);
  if (b->dev.doms) cudaFree(b->dev.doms);
  if (b->dev.items) cudaFree(b->dev.items);
  if (b->dev.ctr) cudaFree(b->dev.ctr);
  if (b->stream) cudaStreamDestroy(b->stream);
  delete b;
  return HLBM_OK;
}

}  // extern "C"
