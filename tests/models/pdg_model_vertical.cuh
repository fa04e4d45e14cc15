// pdg_model_vertical.cuh -- the smallest models of the problem template of
// Sec. 2 of arXiv 2404.18034, for the tests: a vertical descent,
//   m' = -alpha ||T||,  v' = T_x / m + g_x,
// with the thrust bounds and the dry mass as path constraints (x = (m, v, y));
// with PDG_VERTICAL_NX 2 the mass alone (x = (m, y)).
#pragma once
#ifndef PDG_VERTICAL_NX
#define PDG_VERTICAL_NX 3
#endif

namespace pdg {

constexpr int NX = PDG_VERTICAL_NX;
constexpr int IM = 0, IY = NX - 1;
// compact df/dx: [0] dvdot/dm, [1] dydot/dm
constexpr int SA_A = 2;
#define PDG_MODEL_NU_ALT 4

template <typename R, int NU>
__device__ __forceinline__ void model_eval(const DParams& P, const R* x, const R* u, R* f, R* A, R* Bd) {
  const R m = x[IM], im = R(1) / m, s = u[NU - 1];
  const R nT = sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]), inT = nT > R(0) ? R(1) / nT : R(0);
  R gp[3] = {R(P.m_dry) - m, nT - R(P.T_max), R(P.T_min) - nT};
  R pen = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i) { gp[i] = gp[i] > R(0) ? gp[i] : R(0); pen += gp[i] * gp[i]; }
  R F[NX];
  F[IM] = -R(P.alpha_mdot) * nT;
  if constexpr (NX == 3) F[1] = u[0] * im + R(P.g[0]);
  F[IY] = pen;
#pragma unroll
  for (int i = 0; i < NX; ++i) f[i] = s * F[i];
  A[0] = -s * im * im * u[0];
  A[1] = -R(2) * s * gp[0];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const R t = u[c] * inT;
    Bd[IM * NU + c] = -s * R(P.alpha_mdot) * t;
    if constexpr (NX == 3) Bd[1 * NU + c] = c == 0 ? s * im : R(0);
    Bd[IY * NU + c] = R(2) * s * (gp[1] - gp[2]) * t;
  }
#pragma unroll
  for (int i = 0; i < NX; ++i) Bd[i * NU + NU - 1] = F[i];
}

template <typename R, int NU>
__device__ __forceinline__ void model_jvp(const R* __restrict__ A, const R* __restrict__ Bd, const R* S, int cu, R lam,
                                          R* d) {
  d[IM] = R(0);
  if constexpr (NX == 3) d[1] = A[0] * S[IM];
  d[IY] = A[1] * S[IM];
  if (cu >= 0) {
#pragma unroll
    for (int i = 0; i < NX; ++i) d[i] += lam * Bd[i * NU + cu];
  }
}

template <int NU>
__device__ __forceinline__ void model_vjp(const double* A, const double* Bd, const double* v, double* xb, double* ub) {
  if constexpr (NX == 3) xb[IM] += A[0] * v[1];
  xb[IM] += A[1] * v[IY];
#pragma unroll
  for (int c = 0; c < NU; ++c) {
#pragma unroll
    for (int i = 0; i < NX; ++i) ub[c] += Bd[i * NU + c] * v[i];
  }
}

template <typename R, int NU>
__device__ __forceinline__ void model_init_node(const DParams& P, const R* x0, R t, R* x, R* u) {
  x[IM] = (R(1) - t) * x0[IM] + t * R(0.5) * (x0[IM] + R(P.m_dry));
  if constexpr (NX == 3) x[1] = (R(1) - t) * x0[1] + t * R(P.z_f[1]);
  x[IY] = 0;
#pragma unroll
  for (int c = 0; c < NU; ++c) u[c] = 0;
  u[0] = x[IM] * R(P.g0);
  u[NU - 1] = R(P.tf_guess);
}

}  // namespace pdg
