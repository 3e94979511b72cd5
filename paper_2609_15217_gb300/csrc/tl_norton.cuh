// tl_norton.cuh -- the implicit Norton viscoplastic law of the Newton
// kernels (the law class of Sec. 4.3), shared by the fused per-point kernel
// (Algorithm 2) and the batched, CPU-driven loop (Algorithm 1).
#pragma once
#include <cmath>

#include "tinylu.h"
#include "tinylu_device.cuh"

namespace tl {

struct NortonParams {
    double lambda, mu, two_mu;
    double dtA;     // dt A
    double gfac;    // -dt A m 2 mu
    int m;
};

// Implicit Norton law at one point (J2 flow, isotropic elasticity, Mandel
// notation: xx, yy, zz, sqrt2*xy, sqrt2*xz, sqrt2*yz; theta = 1):
//   sig  = sig0 + lambda tr(de) 1 + 2 mu de,  s = dev sig,
//   seq  = sqrt(3/2 s:s), n = 3/2 s / seq,
//   F_el = de - deps + dp n,  F_p = dp - dt A seq^m,
//   dF_el/dde = I + dp (2 mu / seq)(3/2 K - n n^T),  dF_el/ddp = n,
//   (assembled as one FMA per entry around its constant part, the lower
//   triangle copied from the upper),
//   dF_p/dde  = -dt A m seq^(m-1) 2 mu n^T,          dF_p/ddp = 1.
// The Newton loop is bound by the FP64 pipe, so the square root and 1 / seq
// run on the integer pipe (sqrt_rn, rcp_rn: the same values) and products of
// parameters come with the job: about 55 of 320 FP64 instructions per
// iteration less than with sqrt, a division and every entry of the Jacobian.
__device__ __forceinline__ void norton_stress(const NortonParams &P, const double (&sig0)[6], const double (&x)[7],
                                              double (&sig)[6])
{
    const double tr = x[0] + x[1] + x[2];
#pragma unroll
    for (int i = 0; i < 6; ++i) sig[i] = sig0[i] + P.two_mu * x[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) sig[i] += P.lambda * tr;
}

// Flow direction n, seq^m and the Jacobian at the stress sig and the
// increment dp = x[6].
__device__ __forceinline__ void norton_jacobian(const NortonParams &P, const double (&sig)[6], double dp,
                                                double (&n)[6], double &pw_m, double (&J)[7][7])
{
    const double p3 = (sig[0] + sig[1] + sig[2]) * (1.0 / 3.0);
    double s[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) s[i] = (i < 3) ? sig[i] - p3 : sig[i];
    double ss = 0.0;
#pragma unroll
    for (int i = 0; i < 6; ++i) ss = fma(s[i], s[i], ss);
    const double seq = dev::sqrt_rn(1.5 * ss);
    const double rseq = dev::rcp_rn(seq);
    const double inv = seq > 0.0 ? rseq : 0.0;
    const double f = 1.5 * inv;
#pragma unroll
    for (int i = 0; i < 6; ++i) n[i] = s[i] * f;
    double pw_m1 = 1.0;
    for (int i = 0; i < P.m - 1; ++i) pw_m1 *= seq;
    pw_m = pw_m1 * seq;

    // dF_el/dde = I + c (3/2 K - n n^T) = C_ij - (c n_i) n_j with the
    // constant part C_ij = delta_ij + 3/2 c K_ij: 1 + c on the normal
    // diagonal, -c/2 between normal components, 1 + 3/2 c on the shear
    // diagonal, 0 elsewhere
    const double c = dp * P.two_mu * inv;
    const double c_nn = 1.0 + c, c_no = -0.5 * c, c_ss = fma(1.5, c, 1.0);
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const double cn = c * n[i];
#pragma unroll
        for (int j = i; j < 6; ++j) {
            const double cij = (i < 3 && j < 3) ? (i == j ? c_nn : c_no) : (i == j ? c_ss : 0.0);
            J[i][j] = fma(-cn, n[j], cij);
            J[j][i] = J[i][j];
        }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) J[i][6] = n[i];
    const double g = P.gfac * pw_m1;
#pragma unroll
    for (int j = 0; j < 6; ++j) J[6][j] = g * n[j];
    J[6][6] = 1.0;
}

__device__ __forceinline__ void norton_eval(const NortonParams &P, const double (&sig0)[6],
                                            const double (&deps)[6], const double (&x)[7],
                                            double (&F)[7], double (&J)[7][7], double (&sig)[6])
{
    norton_stress(P, sig0, x, sig);
    double n[6], pw_m;
    norton_jacobian(P, sig, x[6], n, pw_m, J);
#pragma unroll
    for (int i = 0; i < 6; ++i) F[i] = fma(x[6], n[i], x[i] - deps[i]);
    F[6] = fma(-P.dtA, pw_m, x[6]);
}

// Lame constants and step data from a TL_LAW_NORTON descriptor; false when
// the descriptor is invalid (n != 7, E <= 0, nu outside (-1, 1/2), m not an
// integer in 1..64, A or dt not finite).
inline bool norton_params_from_law(const tl_law &law, NortonParams *P)
{
    if (law.id != TL_LAW_NORTON || law.n != 7) return false;
    const double E = law.params[0], nu = law.params[1], Acoef = law.params[2], m = law.params[3],
                 dt = law.params[4];
    if (!(E > 0.0) || !(nu > -1.0 && nu < 0.5) || !(m >= 1.0 && m <= 64.0) || m != std::floor(m) ||
        !std::isfinite(Acoef) || !std::isfinite(dt))
        return false;
    P->lambda = E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu));
    P->mu = E / (2.0 * (1.0 + nu));
    P->two_mu = 2.0 * P->mu;
    P->dtA = dt * Acoef;
    P->gfac = -(dt * Acoef) * m * P->two_mu;
    P->m = static_cast<int>(m);
    return true;
}

template <int N>
__device__ __forceinline__ double norm2(const double (&F)[N])
{
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i) s = fma(F[i], F[i], s);
    return dev::sqrt_rn(s);
}

}  // namespace tl
