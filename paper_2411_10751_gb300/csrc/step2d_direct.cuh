// Fused pull-collide-source step on D2Q37 without staging: every thread pulls
// its node's populations straight into registers.
//
// A block owns the same 32 x 8 tile as the staged kernel (step2d.cuh) with one
// node per thread, and further warps take the nodes of the frame around it (the
// 80 ring nodes of theta for H_i, or the 276 frame nodes of psi for F^SC) at
// the same time: all of a tile's loads are in flight at once, whatever the row
// pitch or the periodic edge, where the staged kernel needs 16-byte aligned
// rows for its TMA boxes and otherwise fills its planes in two to five passes
// per thread.  The frame's lines are the neighbour tiles' (L1 or L2).
// The pseudopotential kind also has a two-launch form (KIND_SCF): psi_kernel
// writes psi of every node, and the step loads it on the tile and its frame, so
// that no frame node's 37 populations are pulled and summed again.
// Node arithmetic, tile and frame are those of the staged kernel, so the
// results are the same bit for bit.
#pragma once

#include "step2d.cuh"

namespace hlbm {

template <int KIND>
struct Direct2 {
  static constexpr int BX = 32, BY = 8, OWN = BX * BY;
  static constexpr int H = KIND == KIND_SC ? 3 : (KIND == KIND_THERMAL ? 1 : 0);
  static constexpr int HF = KIND == KIND_SCF ? 3 : H;   // frame of the neighbour field
  using Fr = Frame2<BX, BY, (HF > 0 ? HF : 1)>;
  static constexpr int FRAME = H > 0 ? Fr::count : 0;
  static constexpr int NT = OWN + (FRAME + 31) / 32 * 32;
};

// psi of this step on the tile and its frame, from the field (KIND_SCF); the
// caller synchronises before reading it
template <class Fr, int HF, int NT>
__device__ __forceinline__ void load_psi_tile(const StepArgs& a, float* aux, int x0, int y0, int tid) {
  for (int k = tid; k < Fr::SW * Fr::SH; k += NT) {
    const int j = k / Fr::SW, i = k - j * Fr::SW;
    const int X = wrap_up(x0 - HF + i, a.nx), Y = wrap_up(y0 - HF + j, a.ny);
    aux[frm<Fr>(k)] = __ldg(a.aux_rd + HLBM_IDX(Y * a.nx + X, a.N, DBG_AUX));
  }
}

// theta or psi of a frame node, from its pulled populations
template <int KIND>
__device__ __forceinline__ float frame_value(const StepArgs& a, float (&g)[37], int node, int y) {
  using L = D2Q37;
  if constexpr (KIND == KIND_SC) {
    float hl;
    const float hd = density_h<L>(g, hl);
    return psi_of<L>(a, hd, hl);
  } else {
    return theta_bar_local<L>(a, g, node, y);
  }
}

// The step of the tile at (x0, y0) by the block's NT threads; aux: the frame
// array in shared memory (free once every thread has returned).  Where NT has no
// room for the frame beside the tile (the batched step's pseudopotential tiles)
// all threads take the frame's nodes first.
template <int ST, int KIND, int NT>
__device__ __forceinline__ void direct_tile(const StepArgs& a, float* aux, int x0, int y0) {
  using C = Codec<ST>;
  using T = typename C::T;
  using L = D2Q37;
  using D = Direct2<KIND>;
  using Fr = typename D::Fr;
  constexpr int BX = D::BX, H = D::H;
  constexpr float Dc = (float)(2.0 * L::cs2);
  constexpr float inv_c0 = (float)(1.0 / L::c0);
  const int nx = a.nx, ny = a.ny, tid = threadIdx.x;
  constexpr bool BESIDE = D::OWN + D::FRAME <= NT;
  const T* fin = static_cast<const T*>(a.fin);
  const bool own = tid < D::OWN;
  float g[37];
  if constexpr (!BESIDE) {
    for (int k = tid; k < D::FRAME; k += NT) {
      int fi, fj;
      Fr::pos(k, fi, fj);
      const int fx = wrap_up(x0 - H + fi, nx), fy = wrap_up(y0 - H + fj, ny);
      gather<L, C>(fin, a.N, nx, ny, 1, fx, fy, 0, g);
      aux[frm<Fr>(fj * Fr::SW + fi)] = frame_value<KIND>(a, g, fy * nx + fx, fy);
    }
    if (!own) {
      __syncthreads();
      return;
    }
  }
  // region coordinates of this thread's node
  int i = (tid & (BX - 1)) + H, j = tid / BX + H;
  if constexpr (H > 0 && BESIDE)
    if (!own) Fr::pos(min(tid - D::OWN, D::FRAME - 1), i, j);
  const int xr = x0 - H + i, yr = y0 - H + j;
  const int x = wrap_up(xr, nx), y = wrap_up(yr, ny), node = y * nx + x;
  const bool active = own && xr < nx && yr < ny;
  if (H == 0 && !own) return;
  if constexpr (KIND == KIND_SCF) load_psi_tile<Fr, D::HF, D::OWN>(a, aux, x0, y0, tid);
  gather<L, C>(fin, a.N, nx, ny, 1, x, y, 0, g);
  if constexpr (H > 0 && BESIDE) {
    if (!own) {
      if (tid - D::OWN < D::FRAME) aux[frm<Fr>(j * Fr::SW + i)] = frame_value<KIND>(a, g, node, y);
      __syncthreads();
      return;
    }
  }
  float dr, dr_l, acc, J[3], Pih;
  moments_h<L>(g, dr, dr_l, acc, J, Pih);
  const float rho = vadd(a.rho0, dr);
  float ga[3];
  accel<2>(a, node, y, ga);
  float Fx = vmul(rho, ga[0]), Fy = vmul(rho, ga[1]), sigma = 0.f;
  const float* ap = aux + (j + D::HF - H) * Fr::SW + i + D::HF - H;
  if constexpr (KIND == KIND_SC || KIND == KIND_SCF) {
    if constexpr (KIND == KIND_SC) aux[frm<Fr>(j * Fr::SW + i)] = psi_of<L>(a, dr, dr_l);
    __syncthreads();
    const float psi = ap[0];
    // F^SC = -G psi(x) sum_i w_i psi(x + c_i) c_i with G = -1
    float sx = 0.f, sy = 0.f;
    static_for<L::NPAIR>([&](auto P) {
      constexpr int q = 2 * P + 1;
      constexpr int cx = L::c(q, 0), cy = L::c(q, 1);
      const float dpsi = ap[cy * Fr::SW + cx] - ap[-cy * Fr::SW - cx];
      if constexpr (cx != 0) sx = vfma((float)(L::w(q) * cx), dpsi, sx);
      if constexpr (cy != 0) sy = vfma((float)(L::w(q) * cy), dpsi, sy);
    });
    const float fsx = vmul(psi, sx), fsy = vmul(psi, sy);
    Fx = vadd(Fx, fsx);
    Fy = vadd(Fy, fsy);
    // P_i trace coefficient (Eq. 3.12): sigma = p_coef |F^SC|^2 / psi^2
    sigma = (psi > 0.f) ? a.p_coef * (fsx * fsx + fsy * fsy) * rcp_nr(psi * psi) : 0.f;
  }
  const float inv_rho = rcp_nr(rho);
  const float ux = vmul(vfma(0.5f, Fx, J[0]), inv_rho), uy = vmul(vfma(0.5f, Fy, J[1]), inv_rho);
  const float uu = vfma(ux, ux, vmul(uy, uy));
  const float G2 = vfma(Dc, sigma, vmul(2.f, vfma(ux, Fx, vmul(uy, Fy))));
  const float tb = vmul(vmul(vfma(0.5f, G2, vsub(Pih, vmul(rho, uu))), inv_rho), 1.f / Dc);
  NodeSrcT<float> s;
  s.hG[0] = s.hG[1] = s.hG[2] = 0.f;
  if constexpr (KIND == KIND_THERMAL) {
    aux[frm<Fr>(j * Fr::SW + i)] = tb;
    __syncthreads();
    const float gtx = 0.5f * (ap[1] - ap[-1]), gty = 0.5f * (ap[Fr::SW] - ap[-Fr::SW]);
    // s^(3) += rho theta (1 - 1/Pr) [delta grad_xi theta], grad_xi = c0 grad
    const float hc = vmul(vmul(rho, vadd(1.f, tb)), a.h_coef * (float)L::c0);
    s.hG[0] = vmul(hc, gtx);
    s.hG[1] = vmul(hc, gty);
  }
  if (!active) return;
  s.dr = 0.f;  // density deviation re-enters in apply_poly_h
  s.rho = rho;
  s.tb = a.isothermal ? 0.f : tb;
  s.u[0] = vmul(ux, inv_c0);
  s.u[1] = vmul(uy, inv_c0);
  s.u[2] = 0.f;
  s.F[0] = vmul(Fx, inv_c0);
  s.F[1] = vmul(Fy, inv_c0);
  s.F[2] = 0.f;
  s.sigma = sigma;
  float K[15];
  poly2<L>(s, a.omega, a.beta, K);
  const float om1 = 1.f - a.omega;
  K[0] = vfma(-om1, acc, K[0]);
  if constexpr (KIND == KIND_SC || KIND == KIND_SCF) K[0] = vadd(K[0], dr_l);
  apply_poly_h<L, 15>(g, K, om1, dr);
  const uint32_t salt = std::is_same<T, float>::value ? 0u : node_salt(node, g[0]);
  if (!HLBM_IN(node, a.N, DBG_STORE)) return;
  T* __restrict__ fout = static_cast<T*>(a.fout) + node;
  static_for<37>([&](auto I) {
    constexpr int q = I;
    fout[(size_t)q * (size_t)a.N] = round_store<T>(g[q], pop_bits(salt, q));
  });
}

// PER: blocks per SM that the registers are sized for
template <int ST, int KIND, int PER>
__global__ void __launch_bounds__(Direct2<KIND>::NT, PER) step2d_direct_kernel(const __grid_constant__ StepArgs a) {
  using D = Direct2<KIND>;
  __shared__ float aux[D::HF > 0 ? D::Fr::SW * D::Fr::SH : 1];
  grid_dependency_wait();
  direct_tile<ST, KIND, D::NT>(a, aux, blockIdx.x * D::BX, blockIdx.y * D::BY);
}

// Blocks per SM that the registers are sized for (us per step): 80 registers
// leave 2 thermal and 3 body-force blocks; one more of each, with 56 and 64
// registers, spills and is slower on small domains and in 16 bits (thermal 64 x 64
// 3.20 / 3.34, 256 x 256 FP16 5.0 / 5.5, 901 x 899 FP16 46.4 / 46.9) but faster on large
// FP32 ones (901 x 899 thermal 55.9 / 51.9, body force 48.9 / 47.9).  The
// pseudopotential block of 17 warps takes 56 registers and 100 B of spills for two
// blocks as soon as the tiles outnumber the SMs (one / two per SM: 256 x 256 7.7 /
// 7.1, 64 x 64 4.0 / 4.3).  Reading psi from its field, three against two: 901 x 899
// 78.0 / 88.4.
template <int KIND>
constexpr int direct2_per_sm() {
  return KIND == KIND_LOCAL || KIND == KIND_SCF ? 3 : 2;
}

template <int ST, int KIND, int PER>
cudaError_t launch_direct2(const StepArgs& a, dim3 grid, cudaStream_t s) {
  return launch_pdl(step2d_direct_kernel<ST, KIND, PER>, grid, Direct2<KIND>::NT, 0, s, a);
}

template <int ST>
cudaError_t launch_direct2_st(const StepArgs& a, int kind, int sms, cudaStream_t s) {
  const dim3 grid((a.nx + 31) / 32, (a.ny + 7) / 8);
  if (kind == KIND_SC)
    return (int)(grid.x * grid.y) <= sms ? launch_direct2<ST, KIND_SC, 1>(a, grid, s)
                                         : launch_direct2<ST, KIND_SC, direct2_per_sm<KIND_SC>()>(a, grid, s);
  if (kind == KIND_SCF) return launch_direct2<ST, KIND_SCF, direct2_per_sm<KIND_SCF>()>(a, grid, s);
  if (kind == KIND_THERMAL) return launch_direct2<ST, KIND_THERMAL, direct2_per_sm<KIND_THERMAL>()>(a, grid, s);
  return launch_direct2<ST, KIND_LOCAL, direct2_per_sm<KIND_LOCAL>()>(a, grid, s);
}

// psi of every node (KIND_SCF): one node per thread, 37 loads and the density's
// sum, so four blocks fit an SM.
template <int ST>
__global__ void __launch_bounds__(256, 4) psi_kernel(const __grid_constant__ StepArgs a) {
  const int x = blockIdx.x * 32 + (threadIdx.x & 31), y = blockIdx.y * 8 + threadIdx.x / 32;
  grid_dependency_wait();
  if (x >= a.nx || y >= a.ny) return;
  float g[37];
  gather<D2Q37, Codec<ST>>(static_cast<const typename Codec<ST>::T*>(a.fin), a.N, a.nx, a.ny, 1, x, y, 0, g);
  const int node = y * a.nx + x;
  a.aux_wr[HLBM_IDX(node, a.N, DBG_AUX)] = frame_value<KIND_SC>(a, g, node, y);
}

}  // namespace hlbm
