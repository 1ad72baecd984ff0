// In-place D2Q37 step (AA pattern) with single-pass neighbour fields: one
// population buffer instead of two, and one read and one write of every
// population per step with no frame of populations.
//
// AA pattern.  Before an even step, slot i of node x holds f_i(x, t) (after
// streaming).  The even step reads node x's own 37 slots, collides, and writes
// f*_i into slot ibar of the same node.  Before an odd step, f_i(x, t) is
// therefore in slot ibar of node x - c_i; the odd step reads those, collides,
// and writes f*_i into slot i of node x + c_i, which is where the next even
// step finds f_i(x + c_i, t + 1).  In both steps the slots a node writes are
// exactly the slots it read (slot i of x + c_i is slot (ibar)bar of
// x - c_ibar), so the update is in place without any ordering between nodes.
//
// Neighbour fields.  grad theta (H_i) and the pseudopotential of F^SC and
// P_i would need the populations of the neighbours at time t, which other
// threads may already have overwritten; they are taken from the previous
// step instead (the single-pass variant of the method): each step writes its
// nodes' theta - 1 (thermal kind) or psi (pseudopotential kind) into one of
// two auxiliary fields and reads the neighbours' from the other.  The frame
// of the auxiliary field (1 or 3 nodes around the 32 x 8 tile) is staged in
// shared memory.
//
// Bytes per node and step: 37 x elem read + 37 x elem write + 4 (own field
// written) + about 4 (the staged field, neighbours served by L2): 304 B FP32.
#include "internal.h"
#include "lattice.cuh"
#include "step2d.cuh"

#include <type_traits>

namespace hlbm {
namespace {

using L = D2Q37;
constexpr int kBX = 32, kBY = 8;

__host__ __device__ constexpr int aa_opp(int i) { return i == 0 ? 0 : (((i - 1) & 1) ? i - 1 : i + 1); }

template <int KIND>
constexpr int frame_of() {
  return KIND == KIND_SC ? 3 : (KIND == KIND_THERMAL ? 1 : 0);
}

// One tile of the step.  ODD: the step's parity; MOM: moments readout (no
// store).  NPT nodes per thread: lane k of thread (tx, ty) is tile row
// ty + k kBY / NPT, and with NPT = 2 the node arithmetic runs on paired FP32
// lanes (float2), rounding exactly like the one-node form.
// aux: the neighbour field on the tile and its frame (shared memory).  sp: null,
// or the tile's populations staged by TMA as Cfg2<ST, KIND_LOCAL> lays them out
// (population i of the tile shifted by -c_i on odd steps) and landed;
// staged_done() is called once they are all in registers (after a barrier where
// they were staged).
template <int ST, int KIND, bool ODD, bool MOM, int NPT, class Done>
__device__ __forceinline__ void aa_tile(const StepArgs& a, float* aux, const typename Codec<ST>::T* sp, int x0, int y0,
                                        Done&& staged_done) {
  using T = typename Codec<ST>::T;
  using V = typename std::conditional<NPT == 2, float2, float>::type;
  using Cf = Cfg2<ST, KIND_LOCAL, false, kBY>;
  constexpr int H = frame_of<KIND>();
  constexpr int SW = kBX + 2 * H, SH = kBY + 2 * H;
  constexpr int TR = kBY / NPT, NT = kBX * TR;   // thread rows, threads
  const int nx = a.nx, ny = a.ny;
  const size_t N = (size_t)a.N;
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kBX + tx;
  const int x = x0 + tx;
  const int xc = x < nx ? x : x % nx;   // inactive lanes still compute (the frame is shared)
  int yck[NPT], nodek[NPT];
  bool activek[NPT];
#pragma unroll
  for (int k = 0; k < NPT; ++k) {
    const int y = y0 + ty + k * TR;
    activek[k] = x < nx && y < ny;
    yck[k] = y < ny ? y : y % ny;
    nodek[k] = yck[k] * nx + xc;
  }

  // the previous step's neighbour field, on the tile and its frame
  if constexpr (H > 0) {
    for (int k = tid; k < SW * SH; k += NT) {
      const int j = k / SW, i = k - j * SW;
      const int X = wrapm(x0 - H + i, nx), Y = wrapm(y0 - H + j, ny);
      aux[k] = __ldg(a.aux_rd + HLBM_IDX((long long)Y * nx + X, a.N, DBG_AUX));
    }
  }
  if (H > 0 || sp) __syncthreads();

  // the nodes' populations at time t
  const T* __restrict__ f = static_cast<const T*>(a.fin);
  V g[37];
  if (sp) {
    static_for<37>([&](auto I) {
      constexpr int i = I;
#pragma unroll
      for (int k = 0; k < NPT; ++k)
        set_lane(g[i], k, to_float(sp[stg<Cf>(i, (ty + k * TR) * Cf::WB + tx + (ODD ? Cf::rem(i) : 0))]));
    });
    __syncthreads();
    staged_done();
  } else {
    int xs[7], ys[NPT][7];
#pragma unroll
    for (int d = -3; d <= 3; ++d) {
      xs[d + 3] = wrap1(xc - d, nx);
#pragma unroll
      for (int k = 0; k < NPT; ++k) ys[k][d + 3] = wrap1(yck[k] - d, ny) * nx;
    }
    static_for<37>([&](auto I) {
      constexpr int i = I;
#pragma unroll
      for (int k = 0; k < NPT; ++k) {
        if constexpr (!ODD) {
          set_lane(g[i], k, to_float((f + (size_t)i * N)[(unsigned)HLBM_IDX(nodek[k], a.N, DBG_GATHER)]));
        } else {
          constexpr int cx = L::c(i, 0), cy = L::c(i, 1), b = aa_opp(i);
          set_lane(g[i], k, to_float((f + (size_t)b * N)[(unsigned)HLBM_IDX(ys[k][cy + 3] + xs[cx + 3], a.N, DBG_GATHER)]));
        }
      }
    });
    staged_done();
  }

  V dr, dr_l, acc, J[3], Pih;
  moments_h<L>(g, dr, dr_l, acc, J, Pih);
  const V rho = vadd(splat<V>(a.rho0), dr);
  V gax, gay;
#pragma unroll
  for (int k = 0; k < NPT; ++k) {
    float ga[3];
    accel<2>(a, nodek[k], yck[k], ga);
    set_lane(gax, k, ga[0]);
    set_lane(gay, k, ga[1]);
  }
  V Fx = vmul(rho, gax), Fy = vmul(rho, gay);
  V sigma = splat<V>(0.f), psi_now = splat<V>(0.f);
  if constexpr (KIND == KIND_SC) {
    // F^SC = -G psi(x) sum_i w_i psi(x + c_i) c_i, G = -1, psi of the previous step
    V sx = splat<V>(0.f), sy = splat<V>(0.f), ps;
    static_for<L::NPAIR>([&](auto P) {
      constexpr int i = 2 * P + 1;
      constexpr int cx = L::c(i, 0), cy = L::c(i, 1);
      V dpsi;
#pragma unroll
      for (int k = 0; k < NPT; ++k) {
        const float* ap = aux + (ty + k * TR + H) * SW + tx + H;
        set_lane(dpsi, k, ap[cy * SW + cx] - ap[-cy * SW - cx]);
      }
      if constexpr (cx != 0) sx = vfma(splat<V>((float)(L::w(i) * cx)), dpsi, sx);
      if constexpr (cy != 0) sy = vfma(splat<V>((float)(L::w(i) * cy)), dpsi, sy);
    });
#pragma unroll
    for (int k = 0; k < NPT; ++k) set_lane(ps, k, aux[(ty + k * TR + H) * SW + tx + H]);
    const V fsx = vmul(ps, sx), fsy = vmul(ps, sy);
    Fx = vadd(Fx, fsx);
    Fy = vadd(Fy, fsy);
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const float p1 = lane(ps, k), f1 = lane(fsx, k), f2 = lane(fsy, k);
      set_lane(sigma, k, (p1 > 0.f) ? a.p_coef * (f1 * f1 + f2 * f2) * rcp_nr(p1 * p1) : 0.f);
      set_lane(psi_now, k, psi_of<L>(a, lane(dr, k), lane(dr_l, k)));
    }
  }
  constexpr float Dc = (float)(2.0 * L::cs2);
  const V inv_rho = vmap(rho, [](float r) { return rcp_nr(r); });
  const V ux = vmul(vfma(splat<V>(0.5f), Fx, J[0]), inv_rho);
  const V uy = vmul(vfma(splat<V>(0.5f), Fy, J[1]), inv_rho);
  const V uu = vfma(ux, ux, vmul(uy, uy));
  const V G2 = vfma(splat<V>(Dc), sigma, vmul(splat<V>(2.f), vfma(ux, Fx, vmul(uy, Fy))));
  const V tb = vmul(vmul(vfma(splat<V>(0.5f), G2, vsub(Pih, vmul(rho, uu))), inv_rho), splat<V>(1.f / Dc));

  if constexpr (MOM) {
    double v[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      if (!activek[k]) continue;
      const int node = nodek[k];
      const float r = lane(rho, k), vx = lane(ux, k), vy = lane(uy, k), t = lane(tb, k);
      if (a.rho_out) a.rho_out[node] = r;
      if (a.u_out) {
        a.u_out[node] = vx;
        a.u_out[N + node] = vy;
      }
      if (a.theta_out) a.theta_out[node] = 1.f + t;
      const bool bad = !(isfinite(r) && r > 0.f && isfinite(vx) && isfinite(vy) && isfinite(t));
      v[0] += lane(dr, k);
      v[1] += (double)r * vx;
      v[2] += (double)r * vy;
      v[4] += 0.5 * ((double)lane(Pih, k) + (double)Dc * lane(dr, k) + 0.5 * (double)lane(G2, k));
      v[5] += bad ? 1.0 : 0.0;
    }
    if (a.partials) {
      __shared__ double red[TR][6];
#pragma unroll
      for (int k = 0; k < 6; ++k)
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
      if (tx == 0)
#pragma unroll
        for (int k = 0; k < 6; ++k) red[ty][k] = v[k];
      __syncthreads();
      if (tid < 6) {
        double sum = 0.0;
        for (int w = 0; w < TR; ++w) sum += red[w][tid];
        a.partials[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 8 + tid] = sum;
      }
    }
    return;
  } else {
    // this step's field for the next step's neighbours
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      if (!activek[k]) continue;
      if constexpr (KIND == KIND_SC) a.aux_wr[nodek[k]] = lane(psi_now, k);
      if constexpr (KIND == KIND_THERMAL) a.aux_wr[nodek[k]] = lane(tb, k);
    }
    NodeSrcT<V> s;
    s.hG[0] = s.hG[1] = s.hG[2] = splat<V>(0.f);
    if constexpr (KIND == KIND_THERMAL) {
      V gtx, gty;
#pragma unroll
      for (int k = 0; k < NPT; ++k) {
        const float* ap = aux + (ty + k * TR + 1) * SW + tx + 1;
        set_lane(gtx, k, 0.5f * (ap[1] - ap[-1]));
        set_lane(gty, k, 0.5f * (ap[SW] - ap[-SW]));
      }
      // s^(3) += rho theta (1 - 1/Pr) [delta grad_xi theta], grad_xi = c0 grad
      const V hc = vmul(vmul(rho, vadd(splat<V>(1.f), tb)), splat<V>(a.h_coef * (float)L::c0));
      s.hG[0] = vmul(hc, gtx);
      s.hG[1] = vmul(hc, gty);
    }
    constexpr float inv_c0 = (float)(1.0 / L::c0);
    s.dr = splat<V>(0.f);
    s.rho = rho;
    s.tb = a.isothermal ? splat<V>(0.f) : tb;
    s.u[0] = vmul(ux, splat<V>(inv_c0));
    s.u[1] = vmul(uy, splat<V>(inv_c0));
    s.u[2] = splat<V>(0.f);
    s.F[0] = vmul(Fx, splat<V>(inv_c0));
    s.F[1] = vmul(Fy, splat<V>(inv_c0));
    s.F[2] = splat<V>(0.f);
    s.sigma = sigma;
    V K[15];
    poly2<L>(s, a.omega, a.beta, K);
    const float om1 = 1.f - a.omega;
    K[0] = vfma(splat<V>(-om1), acc, K[0]);
    if constexpr (KIND == KIND_SC) K[0] = vadd(K[0], dr_l);
    apply_poly_h<L, 15>(g, K, om1, dr);
    T* __restrict__ fo = static_cast<T*>(a.fout);
    // the odd step's store offsets are recomputed here from a copy of x that
    // the compiler cannot match with the load offsets, so that the loads'
    // offset arrays need not stay live across the collision
    int xl = xc;
    asm volatile("" : "+r"(xl));
    int xt[7];
#pragma unroll
    for (int d = -3; d <= 3; ++d) xt[d + 3] = ODD ? wrap1(xl + d, nx) : 0;
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      if (!activek[k] || !HLBM_IN(nodek[k], a.N, DBG_STORE)) continue;
      const int node = nodek[k];
      int yl = yck[k];
      asm volatile("" : "+r"(yl));
      int yt[7];
#pragma unroll
      for (int d = -3; d <= 3; ++d) yt[d + 3] = ODD ? wrap1(yl + d, ny) * nx : 0;
      // 16-bit storage: stochastic rounding keyed by node and result (step_common.cuh)
      const uint32_t salt = std::is_same<T, float>::value ? 0u : node_salt(node, lane(g[0], k));
      static_for<37>([&](auto I) {
        constexpr int i = I;
        constexpr int b = aa_opp(i);
        const T v = round_store<T>(lane(g[i], k), pop_bits(salt, i));
        if constexpr (!ODD) {
          fo[(size_t)b * N + node] = v;                             // slot ibar of x
        } else {
          constexpr int cx = L::c(i, 0), cy = L::c(i, 1);
          const long long o = (long long)i * N + yt[cy + 3] + xt[cx + 3];
          if (HLBM_IN(o, 37 * a.N, DBG_STORE)) fo[o] = v;           // slot i of x + c_i
        }
      });
    }
  }
}

template <int ST, int KIND, bool ODD, bool MOM, int NPT>
__global__ void __launch_bounds__(kBX * kBY / NPT, 2 * NPT) aa_step_kernel(const __grid_constant__ StepArgs a) {
  constexpr int H = frame_of<KIND>();
  __shared__ float aux[(H > 0) ? (kBX + 2 * H) * (kBY + 2 * H) : 1];
  grid_dependency_wait();
  aa_tile<ST, KIND, ODD, MOM, NPT>(a, aux, nullptr, blockIdx.x * kBX, blockIdx.y * kBY, [] {});
}

// Persistent CTAs, two nodes per thread, that stage the next tile's populations
// by TMA while the current one collides (tiles in row-major order from the
// step's never-reset counter, backwards on every other step; tiles whose boxes
// would cross the periodic edge pull as above).  A tile writes only the slots it
// read, so the copies of the next tile wait for nothing; what a box holds beyond
// its tile's slots may be changing meanwhile and is not used.
template <int ST, int KIND>
struct AaRing {
  using Cf = Cfg2<ST, KIND_LOCAL, false, kBY>;
  static constexpr int H = frame_of<KIND>();
  static constexpr int AUX = H > 0 ? ((kBX + 2 * H) * (kBY + 2 * H) * 4 + 127) / 128 * 128 : 0;
  static constexpr int BYTES = Cf::POP_BYTES + AUX + 128;
};

template <int ST, int KIND, bool ODD>
__global__ void __launch_bounds__(kBX * kBY / 2, 4)
    aa_persistent_kernel(const __grid_constant__ StepArgs a, const __grid_constant__ CUtensorMap tmap) {
  using R = AaRing<ST, KIND>;
  using Cf = typename R::Cf;
  using T = typename Codec<ST>::T;
  constexpr int W = kBY / 2;   // warps
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int s_first, s_ahead;
  T* sp = reinterpret_cast<T*>(smem);
  float* aux = reinterpret_cast<float*>(smem + Cf::POP_BYTES);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + Cf::POP_BYTES + R::AUX);
  const int tid = threadIdx.y * kBX + threadIdx.x, warp = threadIdx.y;
  const int ntx = (a.nx + kBX - 1) / kBX, ntiles = ntx * ((a.ny + kBY - 1) / kBY);
  const unsigned long long period = (unsigned long long)ntiles + gridDim.x;
  if (!HLBM_IN(smem_u32(smem) & 127u, 1, DBG_SMEM)) return;   // TMA destinations need 128-byte alignment
  auto origin = [&](int t, int& x0, int& y0) {
    const int u = a.reverse ? ntiles - 1 - t : t;
    const int ty = u / ntx;
    y0 = ty * kBY;
    x0 = (u - ty * ntx) * kBX;
  };
  auto stage = [&](int t) {   // lane 0 of every warp: a share of the planes of tile t
    if (t >= ntiles) return;
    int x0, y0;
    origin(t, x0, y0);
    if (!tile_boxed<Cf>(a, x0, y0)) return;
    fence_proxy_async_smem();
    if (warp == 0) mbar_arrive_expect_tx(bar, Cf::TX_BYTES);
    if (a.debug_skip_tma) return;   // test hook: the wait must expire
    static_for<37>([&](auto I) {
      constexpr int i = I;
      if (i % W != warp) return;
      const int bx = ODD ? x0 - L::c(i, 0) - Cf::rem(i) : x0, by = ODD ? y0 - L::c(i, 1) : y0;
      if (!HLBM_IN(bx % Cf::A, 1, DBG_BOX) || !HLBM_IN(bx, a.nx - Cf::WB + 1, DBG_BOX) ||
          !HLBM_IN(by, a.ny - Cf::HB + 1, DBG_BOX))
        return;   // (debug build) a dropped copy leaves the barrier short
      tma_load_3d(sp + i * Cf::PLANE, &tmap, bx, by, ODD ? aa_opp(i) : i, bar);
    });
  };
  unsigned long long raw = 0;
  grid_dependency_wait();
  if (tid == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
    const int t0 = (int)(atomicAdd(a.tile_ctr, 1ull) % period);
    s_first = t0;
    s_ahead = t0 < ntiles ? (int)(atomicAdd(a.tile_ctr, 1ull) % period) : t0;
  }
  __syncthreads();
  int t = s_first;
  if ((tid & 31) == 0) stage(t);
  uint32_t phase = 0;
  while (t < ntiles) {
    const int tn = s_ahead;
    int x0, y0;
    origin(t, x0, y0);
    const bool boxed = tile_boxed<Cf>(a, x0, y0);
    if (boxed) {
      const bool ok = mbar_wait_bounded(bar, phase, a.wait_ns);
      if (!__syncthreads_and(ok)) {
        if (tid == 0) atomicExch(a.status, (int)5 /* HLBM_ETIMEOUT */);
        mbar_wait_bounded(bar, phase, a.wait_ns);
        __syncthreads();
        return;
      }
      phase ^= 1u;
    }
    aa_tile<ST, KIND, ODD, false, 2>(a, aux, boxed ? sp : nullptr, x0, y0, [&] {
      if ((tid & 31) == 0) stage(tn);
      if (tid == 0 && tn < ntiles) raw = atomicAdd(a.tile_ctr, 1ull);
    });
    __syncthreads();   // every thread has read s_ahead and is done with aux
    if (tid == 0) s_ahead = tn < ntiles ? (int)(raw % period) : tn;
    __syncthreads();
    t = tn;
  }
}

template <int ST, int KIND>
int aa_persistent_ctas() {
  static std::atomic<int> cache[kMaxDevicesCached];
  return per_device_cached(cache, [](int dev) {
    int sms = 0, e = 0, o = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(aa_persistent_kernel<ST, KIND, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, AaRing<ST, KIND>::BYTES);
    cudaFuncSetAttribute(aa_persistent_kernel<ST, KIND, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, AaRing<ST, KIND>::BYTES);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&e, aa_persistent_kernel<ST, KIND, false>, kBX * kBY / 2, AaRing<ST, KIND>::BYTES);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, aa_persistent_kernel<ST, KIND, true>, kBX * kBY / 2, AaRing<ST, KIND>::BYTES);
    const int per = std::min(e, o);   // one grid for both parities: they share the counter's period
    return (sms > 0 ? sms : 1) * (per > 0 ? per : 1);
  });
}

// Initial state in the even layout: slot i of node x = f^eq_i(x); the
// neighbour field the first step reads (theta - 1, or psi of the density).
template <int ST, int KIND>
__global__ void __launch_bounds__(256) aa_init_kernel(const __grid_constant__ StepArgs a, const float* __restrict__ rho,
                                                      const float* __restrict__ u, const float* __restrict__ theta) {
  using T = typename Codec<ST>::T;
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= a.N) return;
  const size_t N = (size_t)a.N;
  NodeSrcT<float> s;
  s.dr = rho[n] - a.rho0;
  s.rho = rho[n];
  s.tb = theta[n] - 1.f;
  constexpr float inv_c0 = (float)(1.0 / L::c0);
  s.u[0] = u[n] * inv_c0;
  s.u[1] = u[N + n] * inv_c0;
  s.u[2] = 0.f;
  s.F[0] = s.F[1] = s.F[2] = 0.f;
  s.hG[0] = s.hG[1] = s.hG[2] = 0.f;
  s.sigma = 0.f;
  float g[37], K[15];
#pragma unroll
  for (int i = 0; i < 37; ++i) g[i] = 0.f;
  poly2<L>(s, 1.f, 0.f, K);
  apply_poly<L, 15>(g, K, 0.f);
  T* __restrict__ fo = static_cast<T*>(a.fout);
  static_for<37>([&](auto I) {
    constexpr int i = I;
    Codec<ST>::st(fo + (size_t)i * N + n, g[i]);
  });
  if constexpr (KIND == KIND_THERMAL) a.aux_wr[n] = theta[n] - 1.f;
  if constexpr (KIND == KIND_SC) a.aux_wr[n] = psi_of<L>(a, rho[n] - a.rho0, 0.f);
}

// steps: two nodes per thread (paired FP32 lanes); the moments readout: one
template <int ST, int KIND>
cudaError_t launch_kind(const StepArgs& a, bool odd, bool mom, const CUtensorMap* tmap, cudaStream_t s) {
  const dim3 grid((a.nx + kBX - 1) / kBX, (a.ny + kBY - 1) / kBY);
  if (mom) {
    const dim3 block(kBX, kBY);
    if (odd) aa_step_kernel<ST, KIND, true, true, 1><<<grid, block, 0, s>>>(a);
    else aa_step_kernel<ST, KIND, false, true, 1><<<grid, block, 0, s>>>(a);
  } else {
    const dim3 block(kBX, kBY / 2);
    if (tmap) {
      const dim3 ctas(std::min((int)(grid.x * grid.y), aa_persistent_ctas<ST, KIND>()));
      return odd ? launch_pdl(aa_persistent_kernel<ST, KIND, true>, ctas, block, AaRing<ST, KIND>::BYTES, s, a, *tmap)
                 : launch_pdl(aa_persistent_kernel<ST, KIND, false>, ctas, block, AaRing<ST, KIND>::BYTES, s, a, *tmap);
    }
    return odd ? launch_pdl(aa_step_kernel<ST, KIND, true, false, 2>, grid, block, 0, s, a)
               : launch_pdl(aa_step_kernel<ST, KIND, false, false, 2>, grid, block, 0, s, a);
  }
  return cudaGetLastError();
}

template <int ST>
cudaError_t launch_st(const StepArgs& a, int kind, bool odd, bool mom, const CUtensorMap* tmap, cudaStream_t s) {
  if (kind == KIND_SC) return launch_kind<ST, KIND_SC>(a, odd, mom, tmap, s);
  if (kind == KIND_THERMAL) return launch_kind<ST, KIND_THERMAL>(a, odd, mom, tmap, s);
  return launch_kind<ST, KIND_LOCAL>(a, odd, mom, tmap, s);
}

template <int ST>
cudaError_t init_st(const StepArgs& a, int kind, const float* rho, const float* u, const float* theta,
                    cudaStream_t s) {
  const unsigned blocks = (unsigned)((a.N + 255) / 256);
  if (kind == KIND_SC) aa_init_kernel<ST, KIND_SC><<<blocks, 256, 0, s>>>(a, rho, u, theta);
  else if (kind == KIND_THERMAL) aa_init_kernel<ST, KIND_THERMAL><<<blocks, 256, 0, s>>>(a, rho, u, theta);
  else aa_init_kernel<ST, KIND_LOCAL><<<blocks, 256, 0, s>>>(a, rho, u, theta);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_aa(const StepArgs& a, int kind, int storage, bool odd, bool mom, const CUtensorMap* tmap,
                      cudaStream_t s) {
  switch (storage) {
    case ST_F32: return launch_st<ST_F32>(a, kind, odd, mom, tmap, s);
    case ST_F16: return launch_st<ST_F16>(a, kind, odd, mom, tmap, s);
    default: return launch_st<ST_BF16>(a, kind, odd, mom, tmap, s);
  }
}

cudaError_t launch_aa_init(const StepArgs& a, int kind, int storage, const float* rho, const float* u,
                           const float* theta, cudaStream_t s) {
  switch (storage) {
    case ST_F32: return init_st<ST_F32>(a, kind, rho, u, theta, s);
    case ST_F16: return init_st<ST_F16>(a, kind, rho, u, theta, s);
    default: return init_st<ST_BF16>(a, kind, rho, u, theta, s);
  }
}

}  // namespace hlbm
