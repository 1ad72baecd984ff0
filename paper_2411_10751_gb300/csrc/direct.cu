// D2Q37 step kernels without staging (step2d_direct.cuh), every storage type,
// and the rule that picks them.
#include "step2d_direct.cuh"

namespace hlbm {
namespace {
int sm_count() {
  static std::atomic<int> cache[kMaxDevicesCached];
  return per_device_cached(cache, [](int dev) {
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
  });
}
}  // namespace

// Without TMA (row pitch not a multiple of 16 bytes) the staged kernel fills
// its planes by per-node gathers and the direct one is faster at every size and
// kind measured (901 x 899, FP32 / FP16 us per step: body force 54.5 -> 47.3 /
// 44.2 -> 39.5, thermal 68.5 -> 58.2 / 54.9 -> 54.1, pseudopotential 113 -> 84.7
// / 93.2 -> 79.2).  With TMA it is faster as long as its blocks fit the device at
// once, where the latency of a step counts (64 x 64: 4.3 -> 3.0, 5.2 -> 3.5, 8.1
// -> 4.4; 256 x 256: 5.5 -> 4.9, 6.7 -> 5.7, 10.1 -> 8.3), and slower beyond
// (384 x 384 body force 7.2 against 8.0, 320 x 320 thermal 7.5 against 8.3,
// 448 x 448 pseudopotential FP16 20.1 against 24.1).
bool direct_d2q37(int kind, int nx, int ny, bool tma) {
  if (!tma) return true;
  const long long tiles = (long long)((nx + 31) / 32) * ((ny + 7) / 8);
  const int per = kind == KIND_SC        ? direct2_per_sm<KIND_SC>()
                  : kind == KIND_THERMAL ? direct2_per_sm<KIND_THERMAL>()
                                         : direct2_per_sm<KIND_LOCAL>();
  return tiles <= (long long)per * sm_count();
}

cudaError_t launch_direct_d2q37(const StepArgs& a, int kind, int storage, cudaStream_t s) {
  switch (storage) {
    case ST_F32: return launch_direct2_st<ST_F32>(a, kind, sm_count(), s);
    case ST_F16: return launch_direct2_st<ST_F16>(a, kind, sm_count(), s);
    default: return launch_direct2_st<ST_BF16>(a, kind, sm_count(), s);
  }
}
}  // namespace hlbm
