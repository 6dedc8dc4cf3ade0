// Zero-order-hold discretisation of one diagonal state (Sec. III-B, Eq. 3) and its adjoint, in double precision.
#pragma once

#include "common.cuh"

namespace ssm {

// exp(z) - 1 for z = a + ib without cancellation near z = 0.
__device__ __forceinline__ void expm1_complex(double a, double b, double& re, double& im) {
    double sb, cb;
    sincos(b, &sb, &cb);
    double sh = sin(0.5 * b);
    re = expm1(a) * cb - 2.0 * sh * sh;
    im = exp(a) * sb;
}

struct ZohTerms {
    double ar, ai;  // Abar = exp(Lambda Delta)
    double gr, gi;  // gamma = (Abar - 1) / Lambda
};

__device__ __forceinline__ ZohTerms zoh_terms(float2 lam, float dt) {
    double lr = lam.x, li = lam.y, d = dt;
    double er, ei;
    expm1_complex(lr * d, li * d, er, ei);
    double n = lr * lr + li * li;
    ZohTerms z;
    z.ar = er + 1.0;
    z.ai = ei;
    z.gr = (er * lr + ei * li) / n;
    z.gi = (ei * lr - er * li) / n;
    return z;
}

// Adjoint of the discretisation for one state: from gAbar and g_gamma (= sum_h conj(B) gBbar).
__device__ __forceinline__ void zoh_adjoint(const ZohTerms& z, float2 lam, float dt, double gar, double gai, double ggr,
                                            double ggi, float2& dLambda, float& dDelta) {
    const double lr = lam.x, li = lam.y, d = dt;
    // dgamma/dLambda = (Delta Abar - gamma) / Lambda     (= (Delta Abar Lambda - (Abar-1)) / Lambda^2)
    const double nr = d * z.ar - z.gr, ni = d * z.ai - z.gi;
    const double n = lr * lr + li * li;
    const double qr = (nr * lr + ni * li) / n, qi = (ni * lr - nr * li) / n;
    // dLambda = conj(Delta Abar) gAbar + conj(dgamma/dLambda) g_gamma
    const double outr = d * (z.ar * gar + z.ai * gai) + (qr * ggr + qi * ggi);
    const double outi = d * (z.ar * gai - z.ai * gar) + (qr * ggi - qi * ggr);
    dLambda = make_float2((float)outr, (float)outi);
    // dDelta = Re(conj(Lambda Abar) gAbar) + Re(conj(Abar) g_gamma)
    const double lar = lr * z.ar - li * z.ai, lai = lr * z.ai + li * z.ar;
    dDelta = (float)((lar * gar + lai * gai) + (z.ar * ggr + z.ai * ggi));
}

}  // namespace ssm
