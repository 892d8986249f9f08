// Adjoint of the RPY mobility product (differentiable form of Mdot, Sec. 3.2).
//
// For L = sum_i G_i.u_i + H_i.w_i with [u; w] = M(X) [F; T]:
//   dL/dF = (M [G; H])_u,  dL/dT = (M [G; H])_w      (M is symmetric)
//   dL/dx_i = sum_j grad_d Phi_ij(d),  d = x_i - x_j, with
//   Phi_ij = G_i.tt(d)F_j + F_i.tt(d)G_j + H_i.rr(d)T_j + T_i.rr(d)H_j
//            + g(r) d.(G_i x T_j + H_i x F_j - G_j x T_i - H_j x F_i)
// (tt, rr even in d; the tr/rt coupling odd, hence the signs).  With
// tt = A I + B d d^T and rr = ar I + br d d^T (B, br multiply (d.f) d):
//   grad_d [g.tt f] = (A'/r)(g.f) d + (B'/r)(g.d)(f.d) d + B[(f.d) g + (g.d) f]
//   grad_d [g(r) d.P] = (g'/r)(d.P) d + g P.
// One pass over j per i recomputes every pair term; nothing of size N^2 is
// stored.  The i-side vectors (G_i, F_i, H_i, T_i) multiply sums of scalars
// or vectors accumulated over a tile, so their products are applied once per
// tile.  FP32 partial sums are folded per tile with TwoSum, as in the forward
// kernel.  Units: coefficients in 1/(8 pi eta), applied once per particle.
#include <cuda_runtime.h>

#include <cstdint>

#include "adjoint_common.cuh"
#include "lm_internal.cuh"

namespace lmk {
namespace {


template <typename R, bool ANG>
struct AAcc {
    static constexpr int C = ANG ? 9 : 6;   // dX(3) dF(3) [dT(3)]
    R p[C];                                 // current-tile partials (running sums in shared memory)
    R sG, sF;                               // scalars multiplying G_i, F_i
    R sH, sT;                               // scalars multiplying H_i, T_i
    R gT[3], gF[3], gG[3], gH[3];           // g-weighted sums of j vectors
};

// One pair.  grad = false skips the gradient (r = 0).
template <typename R, bool ANG>
__device__ __forceinline__ void adj_pair(R dx, R dy, R dz, const Coef<R>& c, bool grad,
                                         const typename V4<R>::type& Fj, const typename V4<R>::type& Gj,
                                         const typename V4<R>::type& Tj, const typename V4<R>::type& Hj,
                                         const IData<R, ANG>& I, AAcc<R, ANG>& a) {
    const R b1 = fma(Fj.x, dx, fma(Fj.y, dy, Fj.z * dz));   // F_j.d
    const R b2 = fma(Gj.x, dx, fma(Gj.y, dy, Gj.z * dz));   // G_j.d
    const R Bb2 = c.B * b2;
    // dF += A G_j + B (G_j.d) d
    a.p[3] = fma(Bb2, dx, fma(c.A, Gj.x, a.p[3]));
    a.p[4] = fma(Bb2, dy, fma(c.A, Gj.y, a.p[4]));
    a.p[5] = fma(Bb2, dz, fma(c.A, Gj.z, a.p[5]));
    if (grad) {
        const R a1 = fma(I.G[0], dx, fma(I.G[1], dy, I.G[2] * dz));  // G_i.d
        const R a2 = fma(I.F[0], dx, fma(I.F[1], dy, I.F[2] * dz));  // F_i.d
        const R S1 = fma(I.G[0], Fj.x, fma(I.G[1], Fj.y, fma(I.G[2], Fj.z,
                     fma(I.F[0], Gj.x, fma(I.F[1], Gj.y, I.F[2] * Gj.z)))));
        const R S2 = fma(a1, b1, a2 * b2);
        R cd = fma(c.Ap, S1, c.Bp * S2);
        const R Ba2 = c.B * a2, Ba1 = c.B * a1;
        a.sG = fma(c.B, b1, a.sG);
        a.sF += Bb2;
        if constexpr (ANG) {
            const R e1 = fma(Tj.x, dx, fma(Tj.y, dy, Tj.z * dz));    // T_j.d
            const R e2 = fma(Hj.x, dx, fma(Hj.y, dy, Hj.z * dz));    // H_j.d
            const R c1 = fma(I.H[0], dx, fma(I.H[1], dy, I.H[2] * dz));
            const R c2 = fma(I.T[0], dx, fma(I.T[1], dy, I.T[2] * dz));
            const R R1 = fma(I.H[0], Tj.x, fma(I.H[1], Tj.y, fma(I.H[2], Tj.z,
                         fma(I.T[0], Hj.x, fma(I.T[1], Hj.y, I.T[2] * Hj.z)))));
            const R R2 = fma(c1, e1, c2 * e2);
            cd = fma(c.arp, R1, fma(c.brp, R2, cd));
            // d.P with P = G_i x T_j + H_i x F_j - G_j x T_i - H_j x F_i
            //   = T_j.(d x G_i) + F_j.(d x H_i) + G_j.(d x T_i) + H_j.(d x F_i)
            const R dP =
                Tj.x * (dy * I.G[2] - dz * I.G[1]) + Tj.y * (dz * I.G[0] - dx * I.G[2]) + Tj.z * (dx * I.G[1] - dy * I.G[0]) +
                Fj.x * (dy * I.H[2] - dz * I.H[1]) + Fj.y * (dz * I.H[0] - dx * I.H[2]) + Fj.z * (dx * I.H[1] - dy * I.H[0]) +
                Gj.x * (dy * I.T[2] - dz * I.T[1]) + Gj.y * (dz * I.T[0] - dx * I.T[2]) + Gj.z * (dx * I.T[1] - dy * I.T[0]) +
                Hj.x * (dy * I.F[2] - dz * I.F[1]) + Hj.y * (dz * I.F[0] - dx * I.F[2]) + Hj.z * (dx * I.F[1] - dy * I.F[0]);
            cd = fma(c.gp, dP, cd);
            const R bc2 = c.br * c2, bc1 = c.br * c1;
            a.p[0] = fma(bc2, Hj.x, fma(bc1, Tj.x, a.p[0]));
            a.p[1] = fma(bc2, Hj.y, fma(bc1, Tj.y, a.p[1]));
            a.p[2] = fma(bc2, Hj.z, fma(bc1, Tj.z, a.p[2]));
            a.sH = fma(c.br, e1, a.sH);
            a.sT = fma(c.br, e2, a.sT);
            a.gT[0] = fma(c.g, Tj.x, a.gT[0]); a.gT[1] = fma(c.g, Tj.y, a.gT[1]); a.gT[2] = fma(c.g, Tj.z, a.gT[2]);
            a.gF[0] = fma(c.g, Fj.x, a.gF[0]); a.gF[1] = fma(c.g, Fj.y, a.gF[1]); a.gF[2] = fma(c.g, Fj.z, a.gF[2]);
            a.gG[0] = fma(c.g, Gj.x, a.gG[0]); a.gG[1] = fma(c.g, Gj.y, a.gG[1]); a.gG[2] = fma(c.g, Gj.z, a.gG[2]);
            a.gH[0] = fma(c.g, Hj.x, a.gH[0]); a.gH[1] = fma(c.g, Hj.y, a.gH[1]); a.gH[2] = fma(c.g, Hj.z, a.gH[2]);
        }
        a.p[0] = fma(cd, dx, fma(Ba2, Gj.x, fma(Ba1, Fj.x, a.p[0])));
        a.p[1] = fma(cd, dy, fma(Ba2, Gj.y, fma(Ba1, Fj.y, a.p[1])));
        a.p[2] = fma(cd, dz, fma(Ba2, Gj.z, fma(Ba1, Fj.z, a.p[2])));
    }
    if constexpr (ANG) {
        // dF += g (H_j x d) ; dT += g (G_j x d) + ar H_j + br (H_j.d) d
        const R e2 = fma(Hj.x, dx, fma(Hj.y, dy, Hj.z * dz));
        a.p[3] = fma(c.g, Hj.y * dz - Hj.z * dy, a.p[3]);
        a.p[4] = fma(c.g, Hj.z * dx - Hj.x * dz, a.p[4]);
        a.p[5] = fma(c.g, Hj.x * dy - Hj.y * dx, a.p[5]);
        const R be2 = c.br * e2;
        a.p[6] = fma(be2, dx, fma(c.ar, Hj.x, fma(c.g, Gj.y * dz - Gj.z * dy, a.p[6])));
        a.p[7] = fma(be2, dy, fma(c.ar, Hj.y, fma(c.g, Gj.z * dx - Gj.x * dz, a.p[7])));
        a.p[8] = fma(be2, dz, fma(c.ar, Hj.z, fma(c.g, Gj.x * dy - Gj.y * dx, a.p[8])));
    }
}

// Apply the tile's i-side products to dX and fold into the running sums
// (shared memory, [c][q][tid]).
template <typename R, bool ANG, int NT, int NI>
__device__ __forceinline__ void flush_tile(const IData<R, ANG>& I, AAcc<R, ANG>& a, R* s_hi, R* s_lo, int q) {
#pragma unroll
    for (int q = 0; q < 3; ++q) a.p[q] = fma(a.sG, I.G[q], fma(a.sF, I.F[q], a.p[q]));
    a.sG = a.sF = R(0);
    if constexpr (ANG) {
#pragma unroll
        for (int q = 0; q < 3; ++q) a.p[q] = fma(a.sH, I.H[q], fma(a.sT, I.T[q], a.p[q]));
        a.sH = a.sT = R(0);
        // + G_i x gT + H_i x gF - gG x T_i - gH x F_i
        a.p[0] += (I.G[1] * a.gT[2] - I.G[2] * a.gT[1]) + (I.H[1] * a.gF[2] - I.H[2] * a.gF[1]) -
                  (a.gG[1] * I.T[2] - a.gG[2] * I.T[1]) - (a.gH[1] * I.F[2] - a.gH[2] * I.F[1]);
        a.p[1] += (I.G[2] * a.gT[0] - I.G[0] * a.gT[2]) + (I.H[2] * a.gF[0] - I.H[0] * a.gF[2]) -
                  (a.gG[2] * I.T[0] - a.gG[0] * I.T[2]) - (a.gH[2] * I.F[0] - a.gH[0] * I.F[2]);
        a.p[2] += (I.G[0] * a.gT[1] - I.G[1] * a.gT[0]) + (I.H[0] * a.gF[1] - I.H[1] * a.gF[0]) -
                  (a.gG[0] * I.T[1] - a.gG[1] * I.T[0]) - (a.gH[0] * I.F[1] - a.gH[1] * I.F[0]);
#pragma unroll
        for (int q = 0; q < 3; ++q) a.gT[q] = a.gF[q] = a.gG[q] = a.gH[q] = R(0);
    }
#pragma unroll
    for (int c = 0; c < AAcc<R, ANG>::C; ++c) {
        const int o = (c * NI + q) * NT + threadIdx.x;
        fold(&s_hi[o], &s_lo[o], a.p[c]);
    }
}

template <typename R, bool ANG, int NT, int NI>
constexpr size_t adj_running_bytes() {
    return (size_t)(ANG ? 9 : 6) * NI * NT * sizeof(R) * (sizeof(R) == 4 ? 2 : 1);
}

template <typename R, bool ANG, int NT, int NI>
__global__ void __launch_bounds__(NT) rpy_adjoint_kernel(const typename V4<R>::type* __restrict__ pos4,
                                                         const void* __restrict__ Fp, const void* __restrict__ Tp,
                                                         const void* __restrict__ Gp, const void* __restrict__ Hp,
                                                         int f64, int64_t N, int64_t ntiles, RpyConst<R> k, double c8,
                                                         void* __restrict__ dX, void* __restrict__ dF,
                                                         void* __restrict__ dT, double* __restrict__ partials) {
    using R4 = typename V4<R>::type;
    constexpr int C = AAcc<R, ANG>::C;
    __shared__ R4 sp[NT], sF[NT], sG[NT];
    __shared__ R4 sT[ANG ? NT : 1], sH[ANG ? NT : 1];
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    R* s_hi = reinterpret_cast<R*>(dyn_smem);
    R* s_lo = s_hi + (sizeof(R) == 4 ? C * NI * NT : 0);
    const int tid = threadIdx.x;
    const int64_t i0 = (int64_t)blockIdx.x * (NT * NI);
    int64_t jb, je;
    split_range(N, NT, ntiles, &jb, &je);
    const R pad = (R)kPadCoord;

    IData<R, ANG> I[NI];
    AAcc<R, ANG> a[NI];
#pragma unroll
    for (int q = 0; q < NI; ++q) {
        const int64_t i = i0 + (int64_t)q * NT + tid;
        if (i < N) {
            const R4 p = pos4[i];
            I[q].x = p.x; I[q].y = p.y; I[q].z = p.z;
        } else {
            I[q].x = I[q].y = I[q].z = -pad;
        }
        const int64_t ii = (i < N) ? i : 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            I[q].F[c] = load_elem<R>(Fp, f64, 3 * ii + c);
            I[q].G[c] = load_elem<R>(Gp, f64, 3 * ii + c);
            if constexpr (ANG) {
                I[q].T[c] = load_elem<R>(Tp, f64, 3 * ii + c);
                I[q].H[c] = load_elem<R>(Hp, f64, 3 * ii + c);
            }
        }
#pragma unroll
        for (int c = 0; c < C; ++c) {
            a[q].p[c] = R(0);
            s_hi[(c * NI + q) * NT + tid] = R(0);
            if (sizeof(R) == 4) s_lo[(c * NI + q) * NT + tid] = R(0);
        }
        a[q].sG = a[q].sF = a[q].sH = a[q].sT = R(0);
#pragma unroll
        for (int c = 0; c < 3; ++c) a[q].gT[c] = a[q].gF[c] = a[q].gG[c] = a[q].gH[c] = R(0);
    }

    R4 np, nF, nG, nT, nH;
    auto fetch = [&](int64_t j) {
        const bool in = j < je;
        if (in) np = pos4[j]; else { np.x = pad; np.y = pad; np.z = pad; }
        const int64_t jj = in ? j : 0;
        const R z = R(0);
        nF.x = in ? load_elem<R>(Fp, f64, 3 * jj) : z; nF.y = in ? load_elem<R>(Fp, f64, 3 * jj + 1) : z; nF.z = in ? load_elem<R>(Fp, f64, 3 * jj + 2) : z;
        nG.x = in ? load_elem<R>(Gp, f64, 3 * jj) : z; nG.y = in ? load_elem<R>(Gp, f64, 3 * jj + 1) : z; nG.z = in ? load_elem<R>(Gp, f64, 3 * jj + 2) : z;
        if constexpr (ANG) {
            nT.x = in ? load_elem<R>(Tp, f64, 3 * jj) : z; nT.y = in ? load_elem<R>(Tp, f64, 3 * jj + 1) : z; nT.z = in ? load_elem<R>(Tp, f64, 3 * jj + 2) : z;
            nH.x = in ? load_elem<R>(Hp, f64, 3 * jj) : z; nH.y = in ? load_elem<R>(Hp, f64, 3 * jj + 1) : z; nH.z = in ? load_elem<R>(Hp, f64, 3 * jj + 2) : z;
        }
        np.w = nF.w = nG.w = nT.w = nH.w = z;
    };
    fetch(jb + tid);

    for (int64_t jt = jb; jt < je; jt += NT) {
        sp[tid] = np; sF[tid] = nF; sG[tid] = nG;
        if constexpr (ANG) { sT[tid] = nT; sH[tid] = nH; }
        __syncthreads();
        if (jt + NT < je) fetch(jt + NT + tid);
#pragma unroll 2
        for (int jj = 0; jj < NT; ++jj) {
            const R4 pj = sp[jj];
            const R4 Fj = sF[jj];
            const R4 Gj = sG[jj];
            R4 Tj, Hj;
            if constexpr (ANG) { Tj = sT[jj]; Hj = sH[jj]; } else { Tj = Fj; Hj = Fj; }
            R dx[NI], dy[NI], dz[NI], r2[NI];
            R mn = R(0);
#pragma unroll
            for (int q = 0; q < NI; ++q) {
                dx[q] = I[q].x - pj.x; dy[q] = I[q].y - pj.y; dz[q] = I[q].z - pj.z;
                r2[q] = fma(dx[q], dx[q], fma(dy[q], dy[q], dz[q] * dz[q]));
                mn = (q == 0) ? r2[q] : fmin(mn, r2[q]);
            }
            if (__any_sync(0xffffffffu, mn < k.four_a2)) {
#pragma unroll
                for (int q = 0; q < NI; ++q) {
                    Coef<R> c;
                    const bool g = exact_coef<R, ANG>(r2[q], k, c);
                    adj_pair<R, ANG>(dx[q], dy[q], dz[q], c, g, Fj, Gj, Tj, Hj, I[q], a[q]);
                }
            } else {
#pragma unroll
                for (int q = 0; q < NI; ++q) {
                    Coef<R> c;
                    far_coef<R, ANG>(r2[q], k, c);
                    adj_pair<R, ANG>(dx[q], dy[q], dz[q], c, true, Fj, Gj, Tj, Hj, I[q], a[q]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < NI; ++q) flush_tile<R, ANG, NT, NI>(I[q], a[q], s_hi, s_lo, q);
        __syncthreads();
    }
    const bool direct = (gridDim.y == 1);
#pragma unroll
    for (int q = 0; q < NI; ++q) {
        const int64_t i = i0 + (int64_t)q * NT + tid;
        if (i >= N) continue;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int o = (c * NI + q) * NT + tid;
            const double v = (double)s_hi[o] + (sizeof(R) == 4 ? (double)s_lo[o] : 0.0);
            if (direct) {
                void* out = (c < 3) ? dX : (c < 6 ? dF : dT);
                if (out == nullptr) continue;
                const int64_t idx = 3 * i + (c % 3);
                if (f64) static_cast<double*>(out)[idx] = c8 * v;
                else static_cast<float*>(out)[idx] = (float)(c8 * v);
            } else {
                partials[((int64_t)blockIdx.y * C + c) * N + i] = v;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Packed FP32 adjoint, translation blocks only: two i-particles per f32x2
// instruction (same scheme as the packed forward kernel).  The j-tile holds
// -x_j, F_j and G_j duplicated into both halves of a float2.  Per far-field
// pair (units 1/(8 pi eta)):
//   dF_i += A G_j + B (G_j.d) d
//   dX_i += [A'/r (G_i.F_j + F_i.G_j) + B'/r ((G_i.d)(F_j.d) + (F_i.d)(G_j.d))] d
//           + B (F_i.d) G_j + B (G_i.d) F_j
//           + [B (F_j.d)] G_i + [B (G_j.d)] F_i        (scalars summed per tile)
// with A'/r = -1/r^3 - 3 K1/r^5 and B'/r = -3/r^5 + 5 K2/r^7.  UJ consecutive
// j share one overlap vote, so that the far-field work of UJ j-particles is
// one block of independent instructions.
// ---------------------------------------------------------------------------
// float4 words per j, plain scalars (a j-value enters a packed instruction as
// the same scalar in both lanes): (-x,-y,-z,Fx) (Fy,Fz,Gx,Gy) (Gz,0,0,0)
constexpr int kAdjX2Words = 3;

template <int NT, int NI>
constexpr size_t adj_x2_smem_bytes() {
    return (size_t)kAdjX2Words * NT * sizeof(float4) + adj_running_bytes<float, false, NT, NI>();
}

template <int NT, int NI, int UJ, int MINB = 1>
__global__ void __launch_bounds__(NT, MINB) rpy_adjoint_x2_kernel(const float4* __restrict__ pos4,
                                                            const void* __restrict__ Fp, const void* __restrict__ Gp,
                                                            int f64, int64_t N, int64_t ntiles, RpyConst<float> k,
                                                            double c8, void* __restrict__ dX, void* __restrict__ dF,
                                                            double* __restrict__ partials) {
    static_assert(NI % 2 == 0, "packed form needs an even number of i-particles per thread");
    static_assert(NT % UJ == 0, "the j tile must hold whole groups of UJ");
    constexpr int NP = NI / 2;
    constexpr int C = 6;   // dX(3) dF(3)
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    float4* s_t = reinterpret_cast<float4*>(dyn_smem);
    float* s_hi = reinterpret_cast<float*>(s_t + kAdjX2Words * NT);
    float* s_lo = s_hi + C * NI * NT;
    const int tid = threadIdx.x;
    const int64_t i0 = (int64_t)blockIdx.x * (NT * NI);
    int64_t jb, je;
    split_range(N, NT, ntiles, &jb, &je);
    const float pad = (float)kPadCoord;

    float2 xi[NP], yi[NP], zi[NP], Fi[NP][3], Gi[NP][3];
    float2 p[NP][C], sG[NP], sF[NP];
#pragma unroll
    for (int pp = 0; pp < NP; ++pp) {
        float v[2][9];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t i = i0 + (int64_t)(2 * pp + h) * NT + tid;
            if (i < N) {
                const float4 q = pos4[i];
                v[h][0] = q.x; v[h][1] = q.y; v[h][2] = q.z;
            } else {
                v[h][0] = v[h][1] = v[h][2] = -pad;
            }
            const int64_t ii = (i < N) ? i : 0;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[h][3 + c] = load_elem<float>(Fp, f64, 3 * ii + c);
                v[h][6 + c] = load_elem<float>(Gp, f64, 3 * ii + c);
            }
        }
        xi[pp] = make_float2(v[0][0], v[1][0]);
        yi[pp] = make_float2(v[0][1], v[1][1]);
        zi[pp] = make_float2(v[0][2], v[1][2]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            Fi[pp][c] = make_float2(v[0][3 + c], v[1][3 + c]);
            Gi[pp][c] = make_float2(v[0][6 + c], v[1][6 + c]);
        }
#pragma unroll
        for (int c = 0; c < C; ++c) p[pp][c] = bc2(0.f);
        sG[pp] = sF[pp] = bc2(0.f);
    }
#pragma unroll
    for (int q = 0; q < NI; ++q) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
            s_hi[(c * NI + q) * NT + tid] = 0.f;
            s_lo[(c * NI + q) * NT + tid] = 0.f;
        }
    }
    const float2 K1 = bc2(k.K1), nK2 = bc2(-k.K2), m3K1 = bc2(-3.f * k.K1), K2x5 = bc2(5.f * k.K2);
    const float2 m1 = bc2(-1.f), m3 = bc2(-3.f);

    float4 np;
    float3 nF, nG;
    auto fetch = [&](int64_t j) {
        if (j < je && LM_INBOUNDS(j >= 0 && j < N, 8, j)) {
            np = pos4[j];
            nF = make_float3(load_elem<float>(Fp, f64, 3 * j), load_elem<float>(Fp, f64, 3 * j + 1), load_elem<float>(Fp, f64, 3 * j + 2));
            nG = make_float3(load_elem<float>(Gp, f64, 3 * j), load_elem<float>(Gp, f64, 3 * j + 1), load_elem<float>(Gp, f64, 3 * j + 2));
        } else {
            np = make_float4(pad, pad, pad, 0.f);
            nF = nG = make_float3(0.f, 0.f, 0.f);
        }
    };
    fetch(jb + tid);

    for (int64_t jt = jb; jt < je; jt += NT) {
        s_t[0 * NT + tid] = make_float4(-np.x, -np.y, -np.z, nF.x);
        s_t[1 * NT + tid] = make_float4(nF.y, nF.z, nG.x, nG.y);
        s_t[2 * NT + tid] = make_float4(nG.z, 0.f, 0.f, 0.f);
        __syncthreads();
        if (jt + NT < je) fetch(jt + NT + tid);
        // UJ consecutive j share one overlap vote (more independent work per warp)
#pragma unroll 1
        for (int jj = 0; jj < NT; jj += UJ) {
            float2 dx[UJ][NP], dy[UJ][NP], dz[UJ][NP], r2[UJ][NP];
            float mn;
#pragma unroll
            for (int u = 0; u < UJ; ++u) {
                const float4 w0 = s_t[0 * NT + jj + u];
                const float2 nx = bc2(w0.x), ny = bc2(w0.y), nz = bc2(w0.z);
#pragma unroll
                for (int pp = 0; pp < NP; ++pp) {
                    dx[u][pp] = add2(xi[pp], nx);
                    dy[u][pp] = add2(yi[pp], ny);
                    dz[u][pp] = add2(zi[pp], nz);
                    r2[u][pp] = fma2(dx[u][pp], dx[u][pp], fma2(dy[u][pp], dy[u][pp], mul2(dz[u][pp], dz[u][pp])));
                    const float m2 = fminf(r2[u][pp].x, r2[u][pp].y);
                    mn = (u == 0 && pp == 0) ? m2 : fminf(mn, m2);
                }
            }
            if (__any_sync(0xffffffffu, mn < k.four_a2)) {
#pragma unroll
                for (int u = 0; u < UJ; ++u) {
                    const float4 w0 = s_t[0 * NT + jj + u], w1 = s_t[1 * NT + jj + u];
                    const float4 w2 = s_t[2 * NT + jj + u];
                    const float4 Fj = make_float4(w0.w, w1.x, w1.y, 0.f), Gj = make_float4(w1.z, w1.w, w2.x, 0.f);
#pragma unroll
                    for (int pp = 0; pp < NP; ++pp) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            IData<float, false> I;
                            AAcc<float, false> t;
                            I.x = I.y = I.z = 0.f;
#pragma unroll
                            for (int c = 0; c < 3; ++c) {
                                I.F[c] = h ? Fi[pp][c].y : Fi[pp][c].x;
                                I.G[c] = h ? Gi[pp][c].y : Gi[pp][c].x;
                            }
#pragma unroll
                            for (int c = 0; c < C; ++c) t.p[c] = 0.f;
                            t.sG = t.sF = 0.f;
                            Coef<float> cf;
                            const float ddx = h ? dx[u][pp].y : dx[u][pp].x, ddy = h ? dy[u][pp].y : dy[u][pp].x;
                            const float ddz = h ? dz[u][pp].y : dz[u][pp].x, rr = h ? r2[u][pp].y : r2[u][pp].x;
                            const bool g = exact_coef<float, false>(rr, k, cf);
                            adj_pair<float, false>(ddx, ddy, ddz, cf, g, Fj, Gj, Fj, Fj, I, t);
                            if (h) {
#pragma unroll
                                for (int c = 0; c < C; ++c) p[pp][c].y += t.p[c];
                                sG[pp].y += t.sG;
                                sF[pp].y += t.sF;
                            } else {
#pragma unroll
                                for (int c = 0; c < C; ++c) p[pp][c].x += t.p[c];
                                sG[pp].x += t.sG;
                                sF[pp].x += t.sF;
                            }
                        }
                    }
                }
            } else {
#pragma unroll
                for (int u = 0; u < UJ; ++u) {
                    const float4 w0 = s_t[0 * NT + jj + u], w1 = s_t[1 * NT + jj + u];
                    const float4 w2 = s_t[2 * NT + jj + u];
                    const float2 Fx = bc2(w0.w), Fy = bc2(w1.x), Fz = bc2(w1.y);
                    const float2 Gx = bc2(w1.z), Gy = bc2(w1.w), Gz = bc2(w2.x);
#pragma unroll
                    for (int pp = 0; pp < NP; ++pp) {
                        const float2 ddx = dx[u][pp], ddy = dy[u][pp], ddz = dz[u][pp];
                        const float2 invr = make_float2(rsq_far(r2[u][pp].x), rsq_far(r2[u][pp].y));
                        const float2 invr2 = mul2(invr, invr);
                        const float2 invr3 = mul2(invr2, invr);
                        const float2 invr5 = mul2(invr3, invr2);
                        const float2 A = fma2(K1, invr3, invr);
                        const float2 B = fma2(nK2, invr5, invr3);
                        const float2 Ap = mul2(invr3, fma2(m3K1, invr2, m1));    // -1/r^3 - 3 K1/r^5
                        const float2 Bp = mul2(invr5, fma2(K2x5, invr2, m3));    // -3/r^5 + 5 K2/r^7
                        const float2 b1 = fma2(Fx, ddx, fma2(Fy, ddy, mul2(Fz, ddz)));   // F_j.d
                        const float2 b2 = fma2(Gx, ddx, fma2(Gy, ddy, mul2(Gz, ddz)));   // G_j.d
                        const float2 Bb2 = mul2(B, b2);
                        p[pp][3] = fma2(Bb2, ddx, fma2(A, Gx, p[pp][3]));
                        p[pp][4] = fma2(Bb2, ddy, fma2(A, Gy, p[pp][4]));
                        p[pp][5] = fma2(Bb2, ddz, fma2(A, Gz, p[pp][5]));
                        const float2 a1 = fma2(Gi[pp][0], ddx, fma2(Gi[pp][1], ddy, mul2(Gi[pp][2], ddz)));
                        const float2 a2 = fma2(Fi[pp][0], ddx, fma2(Fi[pp][1], ddy, mul2(Fi[pp][2], ddz)));
                        const float2 S1 = fma2(Gi[pp][0], Fx, fma2(Gi[pp][1], Fy, fma2(Gi[pp][2], Fz,
                                          fma2(Fi[pp][0], Gx, fma2(Fi[pp][1], Gy, mul2(Fi[pp][2], Gz))))));
                        const float2 S2 = fma2(a1, b1, mul2(a2, b2));
                        const float2 cd = fma2(Ap, S1, mul2(Bp, S2));
                        const float2 Ba2 = mul2(B, a2), Ba1 = mul2(B, a1);
                        sG[pp] = fma2(B, b1, sG[pp]);
                        sF[pp] = add2(sF[pp], Bb2);
                        p[pp][0] = fma2(cd, ddx, fma2(Ba2, Gx, fma2(Ba1, Fx, p[pp][0])));
                        p[pp][1] = fma2(cd, ddy, fma2(Ba2, Gy, fma2(Ba1, Fy, p[pp][1])));
                        p[pp][2] = fma2(cd, ddz, fma2(Ba2, Gz, fma2(Ba1, Fz, p[pp][2])));
                    }
                }
            }
        }
        // apply the tile's i-side scalars and fold into the running sums
#pragma unroll
        for (int pp = 0; pp < NP; ++pp) {
#pragma unroll
            for (int c = 0; c < 3; ++c) p[pp][c] = fma2(sG[pp], Gi[pp][c], fma2(sF[pp], Fi[pp][c], p[pp][c]));
            sG[pp] = sF[pp] = bc2(0.f);
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int o0 = (c * NI + 2 * pp) * NT + tid;
                const int o1 = o0 + NT;
                fold(&s_hi[o0], &s_lo[o0], p[pp][c].x);
                fold(&s_hi[o1], &s_lo[o1], p[pp][c].y);
            }
        }
        __syncthreads();
    }
    const bool direct = (gridDim.y == 1);
#pragma unroll
    for (int q = 0; q < NI; ++q) {
        const int64_t i = i0 + (int64_t)q * NT + tid;
        if (i >= N) continue;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int o = (c * NI + q) * NT + tid;
            const double v = (double)s_hi[o] + (double)s_lo[o];
            if (direct) {
                void* out = (c < 3) ? dX : dF;
                if (out == nullptr) continue;
                const int64_t idx = 3 * i + (c % 3);
                if (f64) static_cast<double*>(out)[idx] = c8 * v;
                else static_cast<float*>(out)[idx] = (float)(c8 * v);
            } else {
                partials[((int64_t)blockIdx.y * C + c) * N + i] = v;
            }
        }
    }
}

__global__ void adj_reduce_kernel(const double* __restrict__ partials, int splits, int C, int64_t N, double c8,
                                  void* __restrict__ dX, void* __restrict__ dF, void* __restrict__ dT, int f64) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)C * N) return;
    const int64_t i = e / C;
    const int c = (int)(e - i * C);
    void* out = (c < 3) ? dX : (c < 6 ? dF : dT);
    if (out == nullptr) return;
    double s = 0.0;
    for (int k = 0; k < splits; ++k) s += partials[((int64_t)k * C + c) * N + i];
    const int64_t idx = 3 * i + (c % 3);
    if (f64) static_cast<double*>(out)[idx] = c8 * s;
    else static_cast<float*>(out)[idx] = (float)(c8 * s);
}


template <typename R, bool ANG, int NI>
cudaError_t launch_adj_t(const AdjointArgs& a, cudaStream_t s) {
    constexpr int NT = 128;
    const int64_t nblk = (a.N + NT * NI - 1) / (NT * NI);
    int64_t ntiles = 0;
    const int splits = (int)split_plan(a.N, NT, a.splits, &ntiles);
    if (nblk > 0x7fffffff || splits > 65535) return cudaErrorInvalidConfiguration;
    if (splits > 1 && a.partials == nullptr) return cudaErrorInvalidValue;
    const double c8 = 1.0 / (8.0 * 3.14159265358979323846 * a.eta);
    const RpyConst<R> k = make_rpy_const<R>(a.a);
    dim3 grid((unsigned)nblk, (unsigned)splits);
    constexpr size_t dyn = adj_running_bytes<R, ANG, NT, NI>();
    static std::atomic<unsigned long long> attr_devs{0};  // devices whose limit is raised
    if (cudaError_t e = smem_attr_once(attr_devs, rpy_adjoint_kernel<R, ANG, NT, NI>, dyn)) return e;
    rpy_adjoint_kernel<R, ANG, NT, NI><<<grid, NT, dyn, s>>>(static_cast<const typename V4<R>::type*>(a.pos4), a.F,
                                                       ANG ? a.T : nullptr, a.G, ANG ? a.H : nullptr, a.fp64, a.N,
                                                       ntiles, k, c8, a.dX, a.dF, ANG ? a.dT : nullptr, a.partials);
    cudaError_t err = cudaGetLastError();
    count_launches(1);
    if (err != cudaSuccess || splits == 1) return err;
    constexpr int C = ANG ? 9 : 6;
    const int64_t tot = (int64_t)C * a.N;
    adj_reduce_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(a.partials, splits, C, a.N, c8, a.dX, a.dF,
                                                                     ANG ? a.dT : nullptr, a.fp64);
    count_launches(1);
    return cudaGetLastError();
}

template <int NT, int NI, int UJ>
cudaError_t launch_adj_x2_t(const AdjointArgs& a, cudaStream_t s) {
    const int64_t nblk = (a.N + NT * NI - 1) / (NT * NI);
    int64_t ntiles = 0;
    const int splits = (int)split_plan(a.N, NT, a.splits, &ntiles);
    if (nblk > 0x7fffffff || splits > 65535) return cudaErrorInvalidConfiguration;
    if (splits > 1 && a.partials == nullptr) return cudaErrorInvalidValue;
    const double c8 = 1.0 / (8.0 * 3.14159265358979323846 * a.eta);
    const RpyConst<float> k = make_rpy_const<float>(a.a);
    dim3 grid((unsigned)nblk, (unsigned)splits);
    constexpr size_t dyn = adj_x2_smem_bytes<NT, NI>();
    static std::atomic<unsigned long long> attr_devs{0};  // devices whose limit is raised
    if (cudaError_t e = smem_attr_once(attr_devs, rpy_adjoint_x2_kernel<NT, NI, UJ>, dyn)) return e;
    rpy_adjoint_x2_kernel<NT, NI, UJ><<<grid, NT, dyn, s>>>(static_cast<const float4*>(a.pos4), a.F, a.G, a.fp64, a.N,
                                                        ntiles, k, c8, a.dX, a.dF, a.partials);
    cudaError_t err = cudaGetLastError();
    count_launches(1);
    if (err != cudaSuccess || splits == 1) return err;
    const int64_t tot = 6 * a.N;
    adj_reduce_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(a.partials, splits, 6, a.N, c8, a.dX, a.dF,
                                                                     nullptr, a.fp64);
    count_launches(1);
    return cudaGetLastError();
}

// Packed translation adjoint configurations: threads {128, 256} x ilp {2, 4}
// x j per vote {1, 2} (AdjointArgs::uj).
template <int NT, int NI>
cudaError_t launch_adj_x2_u(const AdjointArgs& a, cudaStream_t s) {
    return a.uj == 2 ? launch_adj_x2_t<NT, NI, 2>(a, s) : launch_adj_x2_t<NT, NI, 1>(a, s);
}

cudaError_t launch_adj_x2(const AdjointArgs& a, cudaStream_t s) {
    if (a.threads == 128 && a.ilp == 2) return launch_adj_x2_u<128, 2>(a, s);
    if (a.threads == 128 && a.ilp == 4) return launch_adj_x2_u<128, 4>(a, s);
    if (a.threads == 256 && a.ilp == 2) return launch_adj_x2_u<256, 2>(a, s);
    if (a.threads == 256 && a.ilp == 4) return launch_adj_x2_u<256, 4>(a, s);
    return cudaErrorInvalidConfiguration;
}

template <int NT, int NI, int UJ>
int adj_x2_occupancy() {
    int n = 0;
    constexpr size_t dyn = adj_x2_smem_bytes<NT, NI>();
    cudaError_t e = cudaFuncSetAttribute(rpy_adjoint_x2_kernel<NT, NI, UJ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)dyn);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, rpy_adjoint_x2_kernel<NT, NI, UJ>, NT, dyn);
    return e == cudaSuccess ? n : 0;
}

}  // namespace

int adjoint_partial_components(int angular) { return angular ? 9 : 6; }

// i-particles per thread: FP32 translation 4 (packed; tunable), FP32 with
// angular blocks 2, FP64 1 (register budget of the heavier angular and FP64
// adjoints).
int adjoint_ilp(int fp64, int angular) { return fp64 ? 1 : (angular ? 2 : 4); }

bool adjoint_config_supported(int fp64, int angular, int threads, int ilp, int uj) {
    if (fp64 || angular) {
        if (uj == 3) return threads == 128 && (fp64 ? ilp == 1 : (ilp == 2 || ilp == 4));   // symmetric scalar form
        if (uj == 4) return !fp64 && threads == 128 && (ilp == 2 || ilp == 4);   // symmetric packed form
        return threads == 128 && ilp == adjoint_ilp(fp64, angular) && uj >= 0 && uj <= 1;
    }
    return (threads == 128 || threads == 256) && (ilp == 2 || ilp == 4) && uj >= 0 && uj <= 3;
}

cudaError_t launch_adjoint(const AdjointArgs& a, cudaStream_t s) {
    if (a.N <= 0) return cudaSuccess;
    if (!adjoint_config_supported(a.fp64, a.angular, a.threads, a.ilp, a.uj)) return cudaErrorInvalidConfiguration;
    if (a.uj >= 3) return launch_adjoint_sym(a, s);
    // one-sided: the scalar kernels for FP64 and for angular blocks
    if (a.fp64 || a.angular) {
        if (a.fp64) return a.angular ? launch_adj_t<double, true, 1>(a, s) : launch_adj_t<double, false, 1>(a, s);
        return launch_adj_t<float, true, 2>(a, s);
    }
    // FP32 translation blocks: the packed (f32x2) kernels
    return launch_adj_x2(a, s);
}

int adjoint_ctas_per_sm(int fp64, int angular, int threads, int ilp, int uj) {
    int n = 0;
    cudaError_t e = cudaErrorInvalidConfiguration;
    if (!adjoint_config_supported(fp64, angular, threads, ilp, uj)) return 0;
#define LM_AOCC(R, ANG, NI)                                                                       \
    {                                                                                             \
        constexpr size_t dyn = adj_running_bytes<R, ANG, 128, NI>();                              \
        e = cudaFuncSetAttribute(rpy_adjoint_kernel<R, ANG, 128, NI>,                             \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);          \
        if (e == cudaSuccess)                                                                     \
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, rpy_adjoint_kernel<R, ANG, 128, NI>, 128, dyn); \
    }
    if (uj >= 3) return adjoint_sym_ctas_per_sm(fp64, angular, threads, ilp, uj);
    if (fp64 && angular) LM_AOCC(double, true, 1)
    else if (fp64) LM_AOCC(double, false, 1)
    else if (angular) LM_AOCC(float, true, 2)
    else {
        const bool two = uj == 2;
        if (threads == 128 && ilp == 2) return two ? adj_x2_occupancy<128, 2, 2>() : adj_x2_occupancy<128, 2, 1>();
        if (threads == 128 && ilp == 4) return two ? adj_x2_occupancy<128, 4, 2>() : adj_x2_occupancy<128, 4, 1>();
        if (threads == 256 && ilp == 2) return two ? adj_x2_occupancy<256, 2, 2>() : adj_x2_occupancy<256, 2, 1>();
        if (threads == 256 && ilp == 4) return two ? adj_x2_occupancy<256, 4, 2>() : adj_x2_occupancy<256, 4, 1>();
        return 0;
    }
#undef LM_AOCC
    return e == cudaSuccess ? n : 0;
}

}  // namespace lmk
