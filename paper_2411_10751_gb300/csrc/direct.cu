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
// 448 x 448 pseudopotential FP16 20.1 against 24.1).  Both sides as of the same
// build; with 32-bit offsets in the pulls the direct side has since gained 5 to
// 20% (64 x 64 body force 2.7, 901 x 899 thermal FP16 46.5, pseudopotential 77.7 /
// 63.0).
bool direct_d2q37(int kind, int nx, int ny, bool tma) {
  if (!tma) return true;
  const long long tiles = (long long)((nx + 31) / 32) * ((ny + 7) / 8);
  const int per = kind == KIND_SC        ? direct2_per_sm<KIND_SC>()
                  : kind == KIND_THERMAL ? direct2_per_sm<KIND_THERMAL>()
                                         : direct2_per_sm<KIND_LOCAL>();
  return tiles <= (long long)per * sm_count();
}

// Two launches read the populations twice but replace the frame's 1.08 pulls
// and psi values per node by one psi value.  They pay off when the tiles exceed
// one wave of blocks and the second read comes from L2 or the rows keep TMA out
// (FP32 us per step, one launch / two: 320 x 320 15.1 / 11.5, 512 x 512 27.4 /
// 23.8, 544 x 544 30.2 / 27.3, 640 x 640 37.8 / 39.2; 641 x 639 46.3 / 41.3, 901 x
// 899 85.3 / 83.5, 1201 x 1199 146.3 / 139.1, FP16 133.9 / 124.4).  Aligned 16-bit
// domains gain nothing (384 x 384 14.3 / 15.0, 512 x 512 23.1 / 23.5).  (Both
// sides of the same build; with 32-bit offsets in the pulls two launches take
// 37.2 at 641 x 639, 77.7 at 901 x 899.)
bool two_launch_d2q37(int storage, int nx, int ny, bool tma) {
  if (direct_d2q37(KIND_SC, nx, ny, true)) return false;   // one wave: a launch more costs more
  return !tma || (storage == ST_F32 && 2.0 * 37 * 4 * (double)nx * ny < 96e6);
}

cudaError_t launch_psi_d2q37(const StepArgs& a, int storage, cudaStream_t s) {
  const dim3 grid((a.nx + 31) / 32, (a.ny + 7) / 8);
  switch (storage) {
    case ST_F32: return launch_pdl(psi_kernel<ST_F32>, grid, dim3(256), 0, s, a);
    case ST_F16: return launch_pdl(psi_kernel<ST_F16>, grid, dim3(256), 0, s, a);
    default: return launch_pdl(psi_kernel<ST_BF16>, grid, dim3(256), 0, s, a);
  }
}

cudaError_t launch_direct_d2q37(const StepArgs& a, int kind, int storage, cudaStream_t s) {
  switch (storage) {
    case ST_F32: return launch_direct2_st<ST_F32>(a, kind, sm_count(), s);
    case ST_F16: return launch_direct2_st<ST_F16>(a, kind, sm_count(), s);
    default: return launch_direct2_st<ST_BF16>(a, kind, sm_count(), s);
  }
}
}  // namespace hlbm
