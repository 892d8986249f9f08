// Device helpers shared by the adjoint kernels, one-sided (adjoint_kernels.cu)
// and symmetric (adjoint_sym_kernels.cu): pair coefficients with their
// derivatives and the i-particle's values.
#pragma once

#include "pair_common.cuh"

namespace lmk {
namespace {

// Coefficients and their derivatives divided by r.
template <typename R>
struct Coef {
    R A, B, g, ar, br;       // values
    R Ap, Bp, gp, arp, brp;  // d/dr divided by r
};

template <typename R, bool ANG>
__device__ __forceinline__ void far_coef(R r2, const RpyConst<R>& k, Coef<R>& c) {
    const R invr = rsq_far(r2);
    const R invr2 = invr * invr;
    const R invr3 = invr2 * invr;
    const R invr5 = invr3 * invr2;
    const R invr7 = invr5 * invr2;
    c.A = fma(k.K1, invr3, invr);
    c.B = fma(-k.K2, invr5, invr3);
    c.Ap = fma(R(-3) * k.K1, invr5, -invr3);
    c.Bp = fma(R(5) * k.K2, invr7, R(-3) * invr5);
    if constexpr (ANG) {
        c.g = invr3;
        c.gp = R(-3) * invr5;
        c.ar = R(-0.5) * invr3;
        c.arp = R(1.5) * invr5;
        c.br = R(1.5) * invr5;
        c.brp = R(-7.5) * invr7;
    }
}

// Exact coefficients; returns false at r = 0 (self / coincident pair), where
// the gradient is taken as zero and only the mobility part contributes.
template <typename R, bool ANG>
__device__ __forceinline__ bool exact_coef(R r2, const RpyConst<R>& k, Coef<R>& c) {
    if (r2 >= k.four_a2) {
        far_coef<R, ANG>(r2, k, c);
        return true;
    }
    const R invr = (r2 > R(0)) ? rsq(r2) : R(0);
    const R r = r2 * invr;
    const R invr3 = invr * invr * invr;
    c.A = k.nA0 - k.nA1 * r;
    c.B = k.nB * invr;
    c.Ap = -k.nA1 * invr;
    c.Bp = -k.nB * invr3;
    if constexpr (ANG) {
        c.g = k.ng0 - k.ng1 * r;
        c.gp = -k.ng1 * invr;
        c.ar = k.inv_a3 * (R(1) - k.rr1 * r + k.rr3 * r * r * r);
        c.arp = k.inv_a3 * (-k.rr1 * invr + R(3) * k.rr3 * r);
        c.br = k.inv_a3 * (k.rrb0 * invr - k.rrb1 * r);
        c.brp = k.inv_a3 * (-k.rrb0 * invr3 - k.rrb1 * invr);
    }
    if (!(r2 > R(0))) {
        c.Ap = c.Bp = R(0);
        if constexpr (ANG) { c.gp = c.arp = c.brp = R(0); }
        return false;
    }
    return true;
}


template <typename R, bool ANG>
struct IData {
    R x, y, z;
    R F[3], G[3];
    R T[ANG ? 3 : 1], H[ANG ? 3 : 1];
};

}  // namespace
}  // namespace lmk
