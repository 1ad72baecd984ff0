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
// kind measured (us per step, staged / direct, 901 x 899, FP32 and FP16: body force
// 54.5 / 48.6, 43.7 / 35.3; thermal 69.1 / 55.9, 53.7 / 46.4; pseudopotential in
// two launches 111 / 77.9, 91.6 / 62.7).  With TMA it is taken as long as its
// blocks fit the device at once, where the latency of a step counts (FP32 64 x 64
// 4.2 / 2.8, 5.1 / 3.2, 8.0 / 4.0; 256 x 256 5.4 / 4.2, 6.8 / 5.1, 9.8 / 7.1).  Just
// beyond, the two are close for the body force (448 x 448 10.2 / 9.8, 544 x 544
// 13.1 / 13.1, FP16 608 x 608 14.9 / 15.7), and the direct one stays ahead for the
// thermal kind up to where its reads stream from HBM (FP32 384 x 384 10.9 / 9.2, 512
// x 512 16.6 / 15.6, 576 x 576 21.1 / 20.4 but 19.3 persistent, 1024 x 1024 55.3
// persistent / 67.4; FP16 320 x 320 7.8 / 7.1, 512 x 512 14.5 / 14.9, 1024 x 1024 45.1 /
// 57.3): the line at one wave is the safe one, not the crossover.
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
// (us per step, staged step / two launches, FP32: 320 x 320 14.8 / 10.2, 512 x 512
// 27.5 / 21.2, 544 x 544 30.3 / 24.2, 768 x 768 54.1 persistent / 52.7, 1024 x 1024
// 89.4 persistent / 93.1; unaligned 641 x 639 60.3 / 37.0, 1201 x 1199 189 / 132).
// In 16 bits aligned rows stay with the staged step, which two launches beat
// up to 608 x 608 (320 x 320 11.7 / 9.9, 512 x 512 22.5 / 20.4, 768 x 768 40.3 / 43.2);
// so they do FP32 a little above the line here (640 x 640 37.5 persistent / 34.8).
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
