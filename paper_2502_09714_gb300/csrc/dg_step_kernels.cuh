// Kernels of one ADER-DG step for the damage rheologies of arXiv 2502.09714
// (CDM of Eq. "cdb-model", IVM of Eq. "ivm-model"; Appendix A), FP32, templated
// on the degree N.
//
//   k_predictor  (dg_predictor.cuh) cell-mean effective Jacobian, Cauchy-Kovalevskaya
//                recursion (Eq. "CKIter-ref-matrix") and damage-rate source at i = 1
//                (Eq. "CKIter-ref-source") -> D, cp, modal traces
//   k_face_flux  (dg_faces.cuh) Rusanov flux (Eq. "rusanov-flux") of every interior
//                face, once per face, time-integrated (the stress at the space-time
//                nodes, the linear terms from the time-integrated trace); absorbing and
//                free-surface fluxes (Appendix A) on boundary faces -> FF, in the
//                face's modal basis
//   k_corrector_tc (dg_corrector.cuh, degrees 2..4) / k_corrector_planes (1, 5): volume flux and damage
//                source (Eqs. "3rd term", "rhs term"), face term (Eq. "2nd
//                term") from FF, update (Eq. "time-integrated")
//
// Each kernel is persistent and walks over tiles of elements (or faces).  The modal
// matrices of the basis are sparse and held in instruction immediates (dg_sparse.cuh).
// For degrees 2..4 the corrector's evaluation at the volume nodes (which feeds the
// pointwise law from tensor memory) and its projection run on the tensor cores
// (tcgen05, TF32 in split parts); the other kernels use the tensor-product structure
// of the rules (planes and rows of nodes).
#pragma once

#include <algorithm>

#include "dg_internal.h"
#include "dg_tc.cuh"

namespace dg {

template <int N>
struct Dim {
  static constexpr int L = n_modes(N), NQ = n_vol_nodes(N), NT = N + 1;
  static constexpr int LP = lp_of(N);
  static constexpr int QS = q_stride(N), DS = d_stride(N), AOFF = d_alpha_offset(N), FFS = ff_stride(N);
};

// Every law's stress has the form sigma = iso delta + sh eps.  CDM (Eq. "cdb-model") and its
// damage rate, with xi = 0 below I2 = 1e-30 and the rate written as C_d gamma_r
// max(0, I1 sqrt(I2) - xi0 I2).
__device__ __forceinline__ void cdm_moduli(const float e[6], float alpha, const MatF& m, float* iso, float* sh,
                                           float* rate) {
  const float I1 = e[0] + e[1] + e[2];
  const float I2 = e[0] * e[0] + e[1] * e[1] + e[2] * e[2] +
                   2.f * (e[3] * e[3] + e[4] * e[4] + e[5] * e[5]);
  // the argument is never denormal where the value is used: the instruction without the scaling
  float rs;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rs) : "f"(I2));
  if (!(I2 > 1e-30f)) rs = 0.f;
  const float s = I2 * rs, xi = I1 * rs;
  const float ag = alpha * m.gamma_r;
  *iso = m.lam0 * I1 - ag * s;
  *sh = fmaf(ag, 2.f * m.xi0 - xi, 2.f * m.mu0);
  *rate = m.cd * m.gamma_r * fmaxf(0.f, I1 * s - m.xi0 * I2);
}

// IVM (Eq. "ivm-model" with l0 = m0 = n0 = 0): sigma = (1 - alpha)(lambda0 I1 delta
// + 2 mu0 eps) and r = (lambda0 I1^2/2 + mu0 I2 - gamma_b (alpha/(1-alpha))^2) /
// (gamma_b tau_b); the material holds gamma_b in gamma_r and 1/(gamma_b tau_b) in cd.
__device__ __forceinline__ void ivm_moduli(const float e[6], float alpha, const MatF& m, float* iso, float* sh,
                                           float* rate) {
  const float I1 = e[0] + e[1] + e[2];
  const float I2 = e[0] * e[0] + e[1] * e[1] + e[2] * e[2] + 2.f * (e[3] * e[3] + e[4] * e[4] + e[5] * e[5]);
  const float f = 1.f - alpha;
  *iso = f * m.lam0 * I1;
  *sh = 2.f * f * m.mu0;
  const float s = alpha / f;
  *rate = m.cd * (0.5f * m.lam0 * I1 * I1 + m.mu0 * I2 - m.gamma_r * s * s);
}

// Nonlinear shear law of the 1-D Riemann verification (Eq. "1d Riemann eqs"):
// sigma = lambda0 I1 delta + 2 mu0 (1 - beta gamma) eps, gamma = sqrt(I2 / 2), which in
// plane shear is sigma_xy = 2 mu0 (1 - beta eps_xy) eps_xy for eps_xy >= 0; beta is
// held in gamma_r and alpha does not evolve.
__device__ __forceinline__ void nlshear_moduli(const float e[6], const MatF& m, float* iso, float* sh, float* rate) {
  const float I1 = e[0] + e[1] + e[2];
  const float I2 = e[0] * e[0] + e[1] * e[1] + e[2] * e[2] + 2.f * (e[3] * e[3] + e[4] * e[4] + e[5] * e[5]);
  *sh = 2.f * m.mu0 * (1.f - m.gamma_r * sqrtf(0.5f * I2));
  *iso = m.lam0 * I1;
  *rate = 0.f;
}

// The pointwise law of the step: 0 = CDM, 1 = IVM, 2 = nonlinear shear.  Every law-
// dependent helper and kernel takes LAW: 0 compiles the CDM alone (the kernels run with
// it whenever the CDM is selected), -1 dispatches on the run-time value `law`.
template <int LAW>
__device__ __forceinline__ void law_moduli(int law, const float e[6], float alpha, const MatF& m, float* iso,
                                           float* sh, float* rate) {
  if constexpr (LAW == 0) {
    cdm_moduli(e, alpha, m, iso, sh, rate);
  } else {
    if (law == 1) ivm_moduli(e, alpha, m, iso, sh, rate);
    else if (law == 2) nlshear_moduli(e, m, iso, sh, rate);
    else cdm_moduli(e, alpha, m, iso, sh, rate);
  }
}

// Effective Lame parameters at a cell mean (CDM: Eq. "effective-cdb" with the sign
// of the xi0 term taken from Eq. "cdb-model"; IVM: Eq. "effective-ivm"; nonlinear
// shear: the secant moduli); q0 holds the ten mode-0 coefficients.
template <int LAW>
__device__ __forceinline__ void effective_lame(int law, const float* q0, const MatF& m, float* lam, float* mu) {
  if constexpr (LAW == 0) law = 0;
  const float r6 = 2.449489742783178f;   // phi_0 = sqrt(6): cell mean = Q_0 sqrt(6)
  if (law == 1) {
    const float f = 1.f - q0[9] * r6;
    *lam = f * m.lam0;
    *mu = f * m.mu0;
    return;
  }
  float u[6];
#pragma unroll
  for (int p = 0; p < 6; ++p) u[p] = q0[p] * r6;
  if (law == 2) {                        // secant moduli of the nonlinear shear law
    const float I2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2] + 2.f * (u[3] * u[3] + u[4] * u[4] + u[5] * u[5]);
    *lam = m.lam0;
    *mu = m.mu0 * (1.f - m.gamma_r * sqrtf(0.5f * I2));
    return;
  }
  const float alpha = q0[9] * r6;
  const float I1 = u[0] + u[1] + u[2];
  const float I2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2] + 2.f * (u[3] * u[3] + u[4] * u[4] + u[5] * u[5]);
  const float xi = I2 > 1e-30f ? I1 * rsqrtf(I2) : 0.f;
  *lam = m.lam0 - alpha * m.gamma_r * xi * (1.f / 3.f);
  *mu = m.mu0 + alpha * m.xi0 * m.gamma_r - 0.5f * alpha * m.gamma_r * xi;
}

// Normal flux on a boundary face (Appendix A, Eqs. "absorbing-flux" and
// "freeSurface-flux") written in global coordinates.  Characteristic analysis
// of the effective isotropic Jacobian along n gives, with the traction
// component sigma_nn = lambda I1 + 2 mu eps_nn, the tangential parts
// v_tan = v - (v.n) n and e_tan = eps n - eps_nn n,
//   a = -v.n + c_p sigma_nn / (lambda + 2 mu),   b = -v_tan / 2 + c_s e_tan:
// free surface (bc 1): strain flux a n n^T + n b^T + b n^T, velocity flux 0
//   (the boundary state is traction free);
// absorbing (bc 2): half that strain flux and the velocity flux
//   ((-sigma_nn / rho + c_p v.n) n + (-2 mu e_tan / rho + c_s v_tan)) / 2
//   (only the outgoing characteristics).
// k_p = c_p / (lambda + 2 mu).  The rotation into the face frame drops out, so
// no tangent vectors are needed.
__device__ __forceinline__ void boundary_flux(int bc, const float u[9], const float n[3], float lam, float mu,
                                              float rho_inv, float cp, float cs, float k_p, float F[9]) {
  const float En[3] = {u[0] * n[0] + u[3] * n[1] + u[5] * n[2], u[3] * n[0] + u[1] * n[1] + u[4] * n[2],
                       u[5] * n[0] + u[4] * n[1] + u[2] * n[2]};
  const float enn = En[0] * n[0] + En[1] * n[1] + En[2] * n[2];
  const float snn = lam * (u[0] + u[1] + u[2]) + 2.f * mu * enn;
  const float vn = u[6] * n[0] + u[7] * n[1] + u[8] * n[2];
  const float a = -vn + k_p * snn;
  float b[3], et[3], vt[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    vt[i] = u[6 + i] - vn * n[i];
    et[i] = En[i] - enn * n[i];
    b[i] = -0.5f * vt[i] + cs * et[i];
  }
  const float h = bc == 2 ? 0.5f : 1.f;
  F[0] = h * (a * n[0] * n[0] + 2.f * n[0] * b[0]);
  F[1] = h * (a * n[1] * n[1] + 2.f * n[1] * b[1]);
  F[2] = h * (a * n[2] * n[2] + 2.f * n[2] * b[2]);
  F[3] = h * (a * n[0] * n[1] + n[0] * b[1] + b[0] * n[1]);
  F[4] = h * (a * n[1] * n[2] + n[1] * b[2] + b[1] * n[2]);
  F[5] = h * (a * n[2] * n[0] + n[2] * b[0] + b[2] * n[0]);
  if (bc == 2) {
    const float pn = 0.5f * (-snn * rho_inv + cp * vn);
#pragma unroll
    for (int i = 0; i < 3; ++i) F[6 + i] = pn * n[i] + 0.5f * (-2.f * mu * et[i] * rho_inv + cs * vt[i]);
  } else {
    F[6] = F[7] = F[8] = 0.f;
  }
}

}  // namespace dg

#include "dg_predictor.cuh"
#include "dg_faces.cuh"
#include "dg_corrector.cuh"
#include "dg_planes.cuh"

namespace dg {

// ---------------------------------------------------------------------------
template <class Cfg, class Kern>
cudaError_t launch_persistent(Kern kern, int64_t tiles, int grid_hint, const StepArgs& a, cudaStream_t s,
                              bool* configured, int* max_blocks, int per_sm = 0) {
  const size_t smem = sizeof(float) * Cfg::SMEM;
  if (!*configured) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    // per_sm given: kernels holding tensor memory, for which the occupancy query does not count by its columns
    if (per_sm == 0) {
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, Cfg::THREADS, smem);
      if (e != cudaSuccess) return e;
    }
    *max_blocks = per_sm > 0 ? per_sm : 1;
    *configured = true;
  }
  int64_t grid = grid_hint > 0 ? static_cast<int64_t>(grid_hint) * *max_blocks : tiles;
  if (grid > tiles) grid = tiles;
  if (grid < 1) grid = 1;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3(static_cast<unsigned>(grid));
  lc.blockDim = dim3(Cfg::THREADS);
  lc.dynamicSmemBytes = smem;
  lc.stream = s;
  lc.attrs = &attr;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, kern, a);
}

template <int N, int LAW, bool TR>
cudaError_t launch_predictor_law(const StepArgs& a, cudaStream_t s) {
  using C = PredCfg<N, TR>;
  static bool cfg = false;
  static int blocks = 1;
  return launch_persistent<C>(k_predictor<N, LAW, TR>, (a.E + C::TE - 1) / C::TE, a.grid_pred > 0 ? a.grid_pred : 148, a,
                              s, &cfg, &blocks);
}

template <int N, int LAW, bool PRE>
cudaError_t launch_faces_law(const StepArgs& a, cudaStream_t s) {
  using C = FaceCfg<N, PRE>;
  static bool cfg[2] = {false, false};
  static int blocks[2] = {1, 1};
  const int grid = a.grid_face > 0 ? a.grid_face : 148;
  // as many rounds over the resident CTAs as whole tiles need, of equal tiles: few faces give every CTA
  // one small tile (384 tets of degree 2: 7.0 us, against 13.4 us with tiles of 21 faces), and the last
  // round is as full as the others (5,184 tets of degree 2: 22.7 -> 20.8 us)
  StepArgs b = a;
  const int64_t slots = static_cast<int64_t>(C::CTAS) * grid, rounds = (a.F + slots * C::TF - 1) / (slots * C::TF);
  b.tile = static_cast<int>(rounds > 0 ? (a.F + slots * rounds - 1) / (slots * rounds) : 1);
  const int64_t tiles = (a.F + b.tile - 1) / b.tile;
  if (a.has_boundary)
    return launch_persistent<C>(k_face_flux<N, LAW, true, PRE>, tiles, grid, b, s, &cfg[1], &blocks[1]);
  return launch_persistent<C>(k_face_flux<N, LAW, false, PRE>, tiles, grid, b, s, &cfg[0], &blocks[0]);
}

// One CTA per SM (a CTA's second team starts on the tiles beyond the grid).
template <int N, int LAW, int TILE>
cudaError_t launch_corrector_tc(const StepArgs& a, int grid, cudaStream_t s) {
  static bool cfg = false;
  static int blocks = 1;
  using C = CorrTcCfg<N, TILE>;
  return launch_persistent<C>(k_corrector_tc<N, LAW, TILE>, (a.E + TILE - 1) / TILE, grid, a, s, &cfg, &blocks, 1);
}

template <int N, int LAW>
cudaError_t launch_corrector_law(const StepArgs& a, cudaStream_t s) {
  const int grid = a.grid_corr > 0 ? a.grid_corr : 148;
  if constexpr (tc_volume(N)) {
    // degree 3: tiles of four elements while each team has at most one (162, 384, 750 tets: 12.3, 12.7, 14.2 us
    // against 15.2, 15.1, 16.0 with eight), else of eight (1,296 and 6,000 tets: 16.9 and 30.8 us against 18.4 and 36.5)
    if constexpr (N == 3) {
      if (a.E <= static_cast<int64_t>(4) * 2 * grid) return launch_corrector_tc<N, LAW, 4>(a, grid, s);
    }
    return launch_corrector_tc<N, LAW, N == 4 ? 4 : 8>(a, grid, s);
  } else {
    static bool cfg = false;
    static int blocks = 1;
    using C = CorrPlaneCfg<N>;
    return launch_persistent<C>(k_corrector_planes<N, LAW>, (a.E + C::TE - 1) / C::TE, grid, a, s, &cfg, &blocks);
  }
}

template <int N, int LAW>
cudaError_t launch_picard_law(const StepArgs& a, cudaStream_t s) {
  using C = PicardCfg<N>;
  static bool cfg = false;
  static int blocks = 1;
  const int grid = a.grid_corr > 0 ? a.grid_corr : 148;
  // few elements: smaller tiles, so that every SM has two
  StepArgs b = a;
  b.tile = static_cast<int>(std::min<int64_t>(C::TE, (a.E + 2 * grid - 1) / (2 * grid)));
  return launch_persistent<C>(k_picard<N, LAW>, (a.E + b.tile - 1) / b.tile, grid, b, s, &cfg, &blocks);
}

// The CDM runs on kernels compiled for it alone; the other laws on the dispatching ones.
template <int N>
cudaError_t launch_predictor_impl(const StepArgs& a, cudaStream_t s) {
  if (a.tr) return a.law == 0 ? launch_predictor_law<N, 0, true>(a, s) : launch_predictor_law<N, -1, true>(a, s);
  return a.law == 0 ? launch_predictor_law<N, 0, false>(a, s) : launch_predictor_law<N, -1, false>(a, s);
}
template <int N>
cudaError_t launch_faces_impl(const StepArgs& a, cudaStream_t s) {
  if (a.tr) return a.law == 0 ? launch_faces_law<N, 0, true>(a, s) : launch_faces_law<N, -1, true>(a, s);
  return a.law == 0 ? launch_faces_law<N, 0, false>(a, s) : launch_faces_law<N, -1, false>(a, s);
}
template <int N>
cudaError_t launch_corrector_impl(const StepArgs& a, cudaStream_t s) {
  return a.law == 0 ? launch_corrector_law<N, 0>(a, s) : launch_corrector_law<N, -1>(a, s);
}
template <int N>
cudaError_t launch_picard_impl(const StepArgs& a, cudaStream_t s) {
  if constexpr (PicardCfg<N>::FITS)
    return a.law == 0 ? launch_picard_law<N, 0>(a, s) : launch_picard_law<N, -1>(a, s);
  return cudaErrorNotSupported;
}

}  // namespace dg

#define DG_INSTANTIATE_STEP(N)                                                                  \
  namespace dg {                                                                                \
  template <> cudaError_t launch_predictor_t<N>(const StepArgs& a, cudaStream_t s) {           \
    return launch_predictor_impl<N>(a, s);                                                      \
  }                                                                                             \
  template <> cudaError_t launch_faces_t<N>(const StepArgs& a, cudaStream_t s) {               \
    return launch_faces_impl<N>(a, s);                                                          \
  }                                                                                             \
  template <> cudaError_t launch_corrector_t<N>(const StepArgs& a, cudaStream_t s) {           \
    return launch_corrector_impl<N>(a, s);                                                      \
  }                                                                                             \
  template <> cudaError_t launch_picard_t<N>(const StepArgs& a, cudaStream_t s) {              \
    return launch_picard_impl<N>(a, s);                                                         \
  }                                                                                             \
  }
