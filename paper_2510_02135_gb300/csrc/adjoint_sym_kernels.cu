// Symmetric adjoint of the mobility product (AdjointArgs::uj 3 and 4): every
// unordered pair {i, j} once, with d = x_i - x_j.  The pair term Phi_ij (top of
// adjoint_kernels.cu) satisfies Phi_ji(-d) = Phi_ij(d), so its gradient g_ij
// goes to dX_i and -g_ij to dX_j; the mobility parts of both directions come
// from the same coefficients (tt and rr even in d, the coupling odd):
//   dF_i += A G_j + B (G_j.d) d + g H_j x d,  dT_i += g G_j x d + ar H_j + br (H_j.d) d
//   dF_j += A G_i + B (G_i.d) d - g H_i x d,  dT_j += -g G_i x d + ar H_i + br (H_i.d) d.
// With P = G_i x T_j + H_i x F_j + T_i x G_j + F_i x H_j and
// cd = (A'/r) S1 + (B'/r) S2 + (ar'/r) R1 + (br'/r) R2 + (g'/r) d.P (S1, S2,
// R1, R2 as in adj_pair):
//   g_ij = cd d + g P + B [(F_j.d) G_i + (G_i.d) F_j + (G_j.d) F_i + (F_i.d) G_j]
//                     + br [(T_j.d) H_i + (H_i.d) T_j + (H_j.d) T_i + (T_i.d) H_j].
// A term that multiplies an i-vector is summed as a scalar over the tile on
// the i-side, one that multiplies a j-vector as a scalar per j on the j-side.
// At r = 0 (self or coincident pairs) the gradient is taken as zero; only the
// mobility parts contribute.
//
// Items, tiles that run one-sided, j-side sums that move over the lanes with
// their j, FP64 slots and their ordered reduction are those of the symmetric
// product (sym_kernels.cu).  The results are bitwise reproducible.
#include <cuda_runtime.h>

#include <cstdint>

#include "adjoint_common.cuh"
#include "sym_common.cuh"

namespace lmk {
namespace {

constexpr int kAdjTileF32 = 128;
constexpr int kAdjTileF64 = 32;

template <bool ANG> constexpr int adj_vals() { return ANG ? 13 : 8; }    // j-side sums per j
template <bool ANG> constexpr int adj_comps() { return ANG ? 9 : 6; }    // dX, dF [, dT]

// Writes the j-side sums of tile t: the warps' rows of s_j added.
template <typename R, int C, int NT, int TJ>
__device__ __forceinline__ void store_j_sums(const R* s_j, const SymGeom& g, int64_t t, int64_t S, bool first,
                                             double* __restrict__ partials) {
    for (int e = threadIdx.x; e < TJ * C; e += NT) {
        const int c = e / TJ, jj = e % TJ;
        const int64_t j = t * TJ + jj;
        if (j >= g.N) continue;
        double s;
        if constexpr (sizeof(R) == 4) {   // a (hi, lo) pair: FP64 operations are dear
            float hi = s_j[c * TJ + jj], lo = 0.f;
#pragma unroll
            for (int w = 1; w < NT / 32; ++w) {
                float x = s_j[(w * C + c) * TJ + jj];
                fold(&hi, &lo, x);
            }
            s = (double)hi + (double)lo;
        } else {
            s = s_j[c * TJ + jj];
#pragma unroll
            for (int w = 1; w < NT / 32; ++w) s += s_j[(w * C + c) * TJ + jj];
        }
        const int64_t o = (S * C + c) * g.N + j;
        // the superblock's slot of j belongs to this item alone; its blocks add in order
        if (LM_INBOUNDS(o < g.slots * C * g.N, 14, o)) partials[o] = first ? s : partials[o] + s;
    }
}

// Writes the i-side running sums of the block at i0 to its slot.
template <typename R, int C, int NT, int NI>
__device__ __forceinline__ void store_i_sums(const R* s_hi, const R* s_lo, const SymGeom& g, int64_t i0, int64_t slot,
                                             double* __restrict__ partials) {
#pragma unroll
    for (int q = 0; q < NI; ++q) {
        const int64_t i = i0 + (int64_t)q * NT + threadIdx.x;
        if (i >= g.N || !LM_INBOUNDS(slot < g.slots, 14, slot)) continue;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int o = (c * NI + q) * NT + threadIdx.x;
            partials[(slot * C + c) * g.N + i] = (double)s_hi[o] + (sizeof(R) == 4 ? (double)s_lo[o] : 0.0);
        }
    }
}

// ---------------------------------------------------------------------------
// Scalar form: FP64, and FP32 with angular blocks.  FP64 is bound by its pipe
// (one warp instruction per 64 cycles and SM quarter).
// ---------------------------------------------------------------------------
template <typename R, bool ANG>
struct SymAcc {
    static constexpr int C = ANG ? 9 : 6;
    R p[C];             // current-tile partials: dX(3) dF(3) [dT(3)]
    R sG, sF, sH, sT;   // scalars multiplying G_i, F_i, H_i, T_i
};

// One pair of the symmetric form: the i-side partials and scalars and, for
// SYM, the j-side sums v = jX(3) jF(3) [jT(3)] then the scalars of F_j, G_j
// [, T_j, H_j].  gg is g where the gradient is taken (r > 0), else 0.
template <typename R, bool ANG, bool SYM>
__device__ __forceinline__ void sym_pair(R dx, R dy, R dz, const Coef<R>& c, R gg, const IData<R, ANG>& I,
                                         const IData<R, ANG>& J, SymAcc<R, ANG>& a, R* v) {
    const R a1 = fma(I.G[0], dx, fma(I.G[1], dy, I.G[2] * dz));   // G_i.d
    const R a2 = fma(I.F[0], dx, fma(I.F[1], dy, I.F[2] * dz));   // F_i.d
    const R b1 = fma(J.F[0], dx, fma(J.F[1], dy, J.F[2] * dz));   // F_j.d
    const R b2 = fma(J.G[0], dx, fma(J.G[1], dy, J.G[2] * dz));   // G_j.d
    const R S1 = fma(I.G[0], J.F[0], fma(I.G[1], J.F[1], fma(I.G[2], J.F[2],
                 fma(I.F[0], J.G[0], fma(I.F[1], J.G[1], I.F[2] * J.G[2])))));
    R cd = fma(c.Ap, S1, c.Bp * fma(a1, b1, a2 * b2));
    const R BA1 = c.B * a1, BA2 = c.B * a2, BB1 = c.B * b1, BB2 = c.B * b2;
    R V[3] = {R(0), R(0), R(0)};
    R rC1 = R(0), rC2 = R(0), rE1 = R(0), rE2 = R(0);
    if constexpr (ANG) {
        const R c1 = fma(I.H[0], dx, fma(I.H[1], dy, I.H[2] * dz));   // H_i.d
        const R c2 = fma(I.T[0], dx, fma(I.T[1], dy, I.T[2] * dz));   // T_i.d
        const R e1 = fma(J.T[0], dx, fma(J.T[1], dy, J.T[2] * dz));   // T_j.d
        const R e2 = fma(J.H[0], dx, fma(J.H[1], dy, J.H[2] * dz));   // H_j.d
        const R R1 = fma(I.H[0], J.T[0], fma(I.H[1], J.T[1], fma(I.H[2], J.T[2],
                     fma(I.T[0], J.H[0], fma(I.T[1], J.H[1], I.T[2] * J.H[2])))));
        // P = G_i x T_j + H_i x F_j + T_i x G_j + F_i x H_j
        R P[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int u = (q + 1) % 3, w = (q + 2) % 3;
            P[q] = fma(I.G[u], J.T[w], fma(-I.G[w], J.T[u], fma(I.H[u], J.F[w], fma(-I.H[w], J.F[u],
                   fma(I.T[u], J.G[w], fma(-I.T[w], J.G[u], fma(I.F[u], J.H[w], -I.F[w] * J.H[u])))))));
        }
        cd = fma(c.arp, R1, fma(c.brp, fma(c1, e1, c2 * e2), fma(c.gp, fma(dx, P[0], fma(dy, P[1], dz * P[2])), cd)));
#pragma unroll
        for (int q = 0; q < 3; ++q) V[q] = gg * P[q];
        rC1 = c.br * c1; rC2 = c.br * c2; rE1 = c.br * e1; rE2 = c.br * e2;
    }
    V[0] = fma(cd, dx, V[0]);
    V[1] = fma(cd, dy, V[1]);
    V[2] = fma(cd, dz, V[2]);
    const R d[3] = {dx, dy, dz};
    // i-side
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        R t = fma(BA2, J.G[q], fma(BA1, J.F[q], V[q]));
        if constexpr (ANG) t = fma(rC2, J.H[q], fma(rC1, J.T[q], t));
        a.p[q] += t;
        a.p[3 + q] = fma(BB2, d[q], fma(c.A, J.G[q], a.p[3 + q]));
    }
    a.sG += BB1;
    a.sF += BB2;
    if constexpr (ANG) {
        a.sH += rE1;
        a.sT += rE2;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int u = (q + 1) % 3, w = (q + 2) % 3;
            // dF_i += g H_j x d ; dT_i += g G_j x d + ar H_j + br (H_j.d) d
            a.p[3 + q] = fma(c.g, fma(J.H[u], d[w], -J.H[w] * d[u]), a.p[3 + q]);
            a.p[6 + q] = fma(rE2, d[q], fma(c.ar, J.H[q], fma(c.g, fma(J.G[u], d[w], -J.G[w] * d[u]), a.p[6 + q])));
        }
    }
    if constexpr (SYM) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            R t = fma(BB2, I.F[q], fma(BB1, I.G[q], V[q]));
            if constexpr (ANG) t = fma(rE2, I.T[q], fma(rE1, I.H[q], t));
            v[q] += t;
            v[3 + q] = fma(BA1, d[q], fma(c.A, I.G[q], v[3 + q]));
        }
        if constexpr (ANG) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int u = (q + 1) % 3, w = (q + 2) % 3;
                // dF_j -= g H_i x d ; dT_j += -g G_i x d + ar H_i + br (H_i.d) d
                v[3 + q] = fma(-c.g, fma(I.H[u], d[w], -I.H[w] * d[u]), v[3 + q]);
                v[6 + q] = fma(rC1, d[q], fma(c.ar, I.H[q], fma(-c.g, fma(I.G[u], d[w], -I.G[w] * d[u]), v[6 + q])));
            }
            v[9] += BA1;    // x F_j
            v[10] += BA2;   // x G_j
            v[11] += rC1;   // x T_j
            v[12] += rC2;   // x H_j
        } else {
            v[6] += BA1;
            v[7] += BA2;
        }
    }
}

template <typename R, bool ANG, int NT, int NI, int TJ>
constexpr size_t adj_sym_s_smem_bytes() {
    return sizeof(R) * ((size_t)(ANG ? 15 : 9) * TJ + (size_t)(NT / 32) * adj_comps<ANG>() * TJ +
                        (size_t)adj_comps<ANG>() * NI * NT * (sizeof(R) == 4 ? 2 : 1));
}

template <typename R, bool ANG, int NT, int NI, int TJ>
__global__ void __launch_bounds__(NT) adj_sym_s_kernel(const typename V4<R>::type* __restrict__ pos4,
                                                       const void* __restrict__ Fp, const void* __restrict__ Tp,
                                                       const void* __restrict__ Gp, const void* __restrict__ Hp,
                                                       int f64, SymGeom g, RpyConst<R> k,
                                                       double* __restrict__ partials) {
    constexpr int C = adj_comps<ANG>(), NV = adj_vals<ANG>(), W = ANG ? 15 : 9;
    extern __shared__ __align__(16) unsigned char adj_sym_smem[];
    R* s_t = reinterpret_cast<R*>(adj_sym_smem);      // [v][jj]: x, F, G, T, H
    R* s_j = s_t + W * TJ;                            // [warp][c][jj]
    R* s_hi = s_j + (NT / 32) * C * TJ;               // [c][q][tid]
    R* s_lo = s_hi + (sizeof(R) == 4 ? C * NI * NT : 0);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const R pad = (R)kPadCoord;
    SymItem it;
    if (!sym_item(g, &it)) return;
    auto value = [&](int64_t i, bool in, int v, R away) -> R {
        if (!in) return v < 3 ? away : R(0);
        if (v < 3) { const typename V4<R>::type p = pos4[i]; return v == 0 ? p.x : (v == 1 ? p.y : p.z); }
        const void* q = v < 6 ? Fp : (v < 9 ? Gp : (v < 12 ? Tp : Hp));
        return load_elem<R>(q, f64, 3 * i + v % 3);
    };
    for (int64_t sub = 0; sub < g.m; ++sub) {
        const int64_t b = it.S * g.m + sub;
        const int64_t i0 = b * (int64_t)(NT * NI);
        if (i0 >= g.N) break;
        IData<R, ANG> I[NI];
        SymAcc<R, ANG> a[NI];
#pragma unroll
        for (int q = 0; q < NI; ++q) {
            const int64_t i = i0 + (int64_t)q * NT + tid;
            const bool in = i < g.N;
            I[q].x = value(i, in, 0, -pad);
            I[q].y = value(i, in, 1, -pad);
            I[q].z = value(i, in, 2, -pad);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                I[q].F[c] = value(i, in, 3 + c, R(0));
                I[q].G[c] = value(i, in, 6 + c, R(0));
                if constexpr (ANG) {
                    I[q].T[c] = value(i, in, 9 + c, R(0));
                    I[q].H[c] = value(i, in, 12 + c, R(0));
                }
            }
            a[q].sG = a[q].sF = a[q].sH = a[q].sT = R(0);
#pragma unroll
            for (int c = 0; c < C; ++c) {
                a[q].p[c] = R(0);
                s_hi[(c * NI + q) * NT + tid] = R(0);
                if (sizeof(R) == 4) s_lo[(c * NI + q) * NT + tid] = R(0);
            }
        }
        const int64_t own = b * g.tb;
        for (int64_t t = it.t0 > own ? it.t0 : own; t < it.t1; ++t) {
            __syncthreads();   // the previous tile's values and sums are no longer read
            for (int e = tid; e < TJ * W; e += NT) {
                const int64_t j = t * TJ + e % TJ;
                s_t[e] = value(j, j < g.N, e / TJ, pad);
            }
            __syncthreads();
            auto load_j = [&](int jj) {
                IData<R, ANG> J;
                J.x = s_t[jj]; J.y = s_t[TJ + jj]; J.z = s_t[2 * TJ + jj];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    J.F[c] = s_t[(3 + c) * TJ + jj];
                    J.G[c] = s_t[(6 + c) * TJ + jj];
                    if constexpr (ANG) {
                        J.T[c] = s_t[(9 + c) * TJ + jj];
                        J.H[c] = s_t[(12 + c) * TJ + jj];
                    }
                }
                return J;
            };
            auto step = [&](auto sym_tag, const IData<R, ANG>& J, R* v) {
                constexpr bool SYM = decltype(sym_tag)::value;
#pragma unroll
                for (int q = 0; q < NI; ++q) {
                    const R dx = I[q].x - J.x, dy = I[q].y - J.y, dz = I[q].z - J.z;
                    const R r2 = fma(dx, dx, fma(dy, dy, dz * dz));
                    Coef<R> c;
                    bool grad = true;
                    if (__any_sync(0xffffffffu, r2 < k.four_a2)) grad = exact_coef<R, ANG>(r2, k, c);
                    else far_coef<R, ANG>(r2, k, c);
                    R gg = R(0);
                    if constexpr (ANG) gg = grad ? c.g : R(0);
                    sym_pair<R, ANG, SYM>(dx, dy, dz, c, gg, I[q], J, a[q], v);
                }
            };
            const bool diag = t < own + g.tb;
            if (diag) {
#pragma unroll 1
                for (int jj = 0; jj < TJ; ++jj) step(BoolTag<false>{}, load_j(jj), nullptr);
            } else {
#pragma unroll 1
                for (int gr = 0; gr < TJ; gr += 32) {
                    R v[NV];
#pragma unroll
                    for (int c = 0; c < NV; ++c) v[c] = R(0);
#pragma unroll 1
                    for (int st = 0; st < 32; ++st) {
                        step(BoolTag<true>{}, load_j(gr + ((lane + st) & 31)), v);
#pragma unroll
                        for (int c = 0; c < NV; ++c) v[c] = __shfl_sync(0xffffffffu, v[c], (lane + 1) & 31);
                    }
                    // home again: dX_j -= vector + scalars x (F_j, G_j [, T_j, H_j])
                    const IData<R, ANG> J = load_j(gr + lane);
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        R x = v[c];
                        if constexpr (ANG)
                            x = fma(v[11], J.T[c], fma(v[12], J.H[c], fma(v[9], J.F[c], fma(v[10], J.G[c], x))));
                        else
                            x = fma(v[6], J.F[c], fma(v[7], J.G[c], x));
                        s_j[(wid * C + c) * TJ + gr + lane] = -x;
                    }
#pragma unroll
                    for (int c = 3; c < C; ++c) s_j[(wid * C + c) * TJ + gr + lane] = v[c];
                }
            }
            // apply the tile's i-side scalars and fold into the running sums
#pragma unroll
            for (int q = 0; q < NI; ++q) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    R x = fma(a[q].sG, I[q].G[c], fma(a[q].sF, I[q].F[c], a[q].p[c]));
                    if constexpr (ANG) x = fma(a[q].sH, I[q].H[c], fma(a[q].sT, I[q].T[c], x));
                    a[q].p[c] = x;
                }
                a[q].sG = a[q].sF = a[q].sH = a[q].sT = R(0);
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const int o = (c * NI + q) * NT + tid;
                    fold(&s_hi[o], &s_lo[o], a[q].p[c]);
                }
            }
            __syncthreads();
            if (!diag) store_j_sums<R, C, NT, TJ>(s_j, g, t, it.S, sub == 0, partials);
        }
        store_i_sums<R, C, NT, NI>(s_hi, s_lo, g, i0, it.S + 1 + it.c, partials);
    }
}

// ---------------------------------------------------------------------------
// Packed FP32 form: two i-particles per f32x2 instruction; the j-words enter
// as the same scalar in both lanes.  Packed operands take no negation, so the
// cross products with d use g d and -g d, and P is formed as the difference of
// its two halves.  j-words: (-x, -y, -z, Fx) (Fy, Fz, Gx, Gy) (Gz, Tx, Ty, Tz)
// (Hx, Hy, Hz, 0), the first three without angular blocks.
// ---------------------------------------------------------------------------
struct PCoef2 {
    float2 A, B, Ap, Bp, g, gp, ar, arp, br, brp;
};

struct Sym6Acc2 {
    float2 p[9];             // dX(3) dF(3) dT(3) of the tile, two i-particles
    float2 sG, sF, sH, sT;   // scalars multiplying G_i, F_i, H_i, T_i
};

// One pair of the packed form: the i-side partials and scalars and, for SYM,
// the j-side sums v: jX(3) jF(3) jT(3), then the scalars of F_j, G_j, T_j, H_j.
template <bool SYM>
__device__ __forceinline__ void sym6_pair2(const float2 (&d)[3], const PCoef2& c, float2 gg, const float2 (&Fi)[3],
                                           const float2 (&Gi)[3], const float2 (&Ti)[3], const float2 (&Hi)[3],
                                           const float* jw, Sym6Acc2& a, float2* v) {
    // j-words: (-x, -y, -z, Fx) (Fy, Fz, Gx, Gy) (Gz, Tx, Ty, Tz) (Hx, Hy, Hz, 0)
    const float* Fj = jw + 3;
    const float* Gj = jw + 6;
    const float* Tj = jw + 9;
    const float* Hj = jw + 12;
    auto doti = [&](const float2 (&w)[3]) { return fma2(w[0], d[0], fma2(w[1], d[1], mul2(w[2], d[2]))); };
    auto dotj = [&](const float* w) { return fma2(bc2(w[0]), d[0], fma2(bc2(w[1]), d[1], mul2(bc2(w[2]), d[2]))); };
    const float2 a1 = doti(Gi), a2 = doti(Fi), c1 = doti(Hi), c2 = doti(Ti);
    const float2 b1 = dotj(Fj), b2 = dotj(Gj), e1 = dotj(Tj), e2 = dotj(Hj);
    const float2 S1 = fma2(Gi[0], bc2(Fj[0]), fma2(Gi[1], bc2(Fj[1]), fma2(Gi[2], bc2(Fj[2]),
                      fma2(Fi[0], bc2(Gj[0]), fma2(Fi[1], bc2(Gj[1]), mul2(Fi[2], bc2(Gj[2])))))));
    const float2 R1 = fma2(Hi[0], bc2(Tj[0]), fma2(Hi[1], bc2(Tj[1]), fma2(Hi[2], bc2(Tj[2]),
                      fma2(Ti[0], bc2(Hj[0]), fma2(Ti[1], bc2(Hj[1]), mul2(Ti[2], bc2(Hj[2])))))));
    // P = G_i x T_j + H_i x F_j + T_i x G_j + F_i x H_j = X - Y
    float2 P[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int u = (q + 1) % 3, w = (q + 2) % 3;
        const float2 X = fma2(Gi[u], bc2(Tj[w]), fma2(Hi[u], bc2(Fj[w]), fma2(Ti[u], bc2(Gj[w]), mul2(Fi[u], bc2(Hj[w])))));
        const float2 Y = fma2(Gi[w], bc2(Tj[u]), fma2(Hi[w], bc2(Fj[u]), fma2(Ti[w], bc2(Gj[u]), mul2(Fi[w], bc2(Hj[u])))));
        P[q] = fma2(bc2(-1.f), Y, X);
    }
    const float2 dP = fma2(d[0], P[0], fma2(d[1], P[1], mul2(d[2], P[2])));
    const float2 cd = fma2(c.Ap, S1, fma2(c.Bp, fma2(a1, b1, mul2(a2, b2)),
                      fma2(c.arp, R1, fma2(c.brp, fma2(c1, e1, mul2(c2, e2)), mul2(c.gp, dP)))));
    const float2 BA1 = mul2(c.B, a1), BA2 = mul2(c.B, a2), BB1 = mul2(c.B, b1), BB2 = mul2(c.B, b2);
    const float2 rC1 = mul2(c.br, c1), rC2 = mul2(c.br, c2), rE1 = mul2(c.br, e1), rE2 = mul2(c.br, e2);
    const float2 ng = mul2(bc2(-1.f), c.g);
    float2 V[3], gd[3], ngd[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        V[q] = fma2(cd, d[q], mul2(gg, P[q]));
        gd[q] = mul2(c.g, d[q]);
        ngd[q] = mul2(ng, d[q]);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int u = (q + 1) % 3, w = (q + 2) % 3;
        a.p[q] = fma2(BA2, bc2(Gj[q]), fma2(BA1, bc2(Fj[q]), fma2(rC2, bc2(Hj[q]), fma2(rC1, bc2(Tj[q]),
                 add2(a.p[q], V[q])))));
        // dF_i += A G_j + B (G_j.d) d + g H_j x d ;  dT_i += g G_j x d + ar H_j + br (H_j.d) d
        a.p[3 + q] = fma2(BB2, d[q], fma2(c.A, bc2(Gj[q]), fma2(bc2(Hj[u]), gd[w], fma2(bc2(Hj[w]), ngd[u],
                     a.p[3 + q]))));
        a.p[6 + q] = fma2(rE2, d[q], fma2(c.ar, bc2(Hj[q]), fma2(bc2(Gj[u]), gd[w], fma2(bc2(Gj[w]), ngd[u],
                     a.p[6 + q]))));
    }
    a.sG = add2(a.sG, BB1);
    a.sF = add2(a.sF, BB2);
    a.sH = add2(a.sH, rE1);
    a.sT = add2(a.sT, rE2);
    if constexpr (SYM) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int u = (q + 1) % 3, w = (q + 2) % 3;
            v[q] = fma2(BB2, Fi[q], fma2(BB1, Gi[q], fma2(rE2, Ti[q], fma2(rE1, Hi[q], add2(v[q], V[q])))));
            // dF_j += A G_i + B (G_i.d) d - g H_i x d ;  dT_j += -g G_i x d + ar H_i + br (H_i.d) d
            v[3 + q] = fma2(BA1, d[q], fma2(c.A, Gi[q], fma2(Hi[u], ngd[w], fma2(Hi[w], gd[u], v[3 + q]))));
            v[6 + q] = fma2(rC1, d[q], fma2(c.ar, Hi[q], fma2(Gi[u], ngd[w], fma2(Gi[w], gd[u], v[6 + q]))));
        }
        v[9] = add2(v[9], BA1);     // x F_j
        v[10] = add2(v[10], BA2);   // x G_j
        v[11] = add2(v[11], rC1);   // x T_j
        v[12] = add2(v[12], rC2);   // x H_j
    }
}

// The same without angular blocks; v = jX(3) jF(3) and the scalars of F_j, G_j.
template <bool SYM>
__device__ __forceinline__ void sym3_pair2(const float2 (&d)[3], const PCoef2& c, const float2 (&Fi)[3],
                                           const float2 (&Gi)[3], const float* jw, Sym6Acc2& a, float2* v) {
    const float* Fj = jw + 3;
    const float* Gj = jw + 6;
    auto doti = [&](const float2 (&w)[3]) { return fma2(w[0], d[0], fma2(w[1], d[1], mul2(w[2], d[2]))); };
    auto dotj = [&](const float* w) { return fma2(bc2(w[0]), d[0], fma2(bc2(w[1]), d[1], mul2(bc2(w[2]), d[2]))); };
    const float2 a1 = doti(Gi), a2 = doti(Fi), b1 = dotj(Fj), b2 = dotj(Gj);
    const float2 S1 = fma2(Gi[0], bc2(Fj[0]), fma2(Gi[1], bc2(Fj[1]), fma2(Gi[2], bc2(Fj[2]),
                      fma2(Fi[0], bc2(Gj[0]), fma2(Fi[1], bc2(Gj[1]), mul2(Fi[2], bc2(Gj[2])))))));
    const float2 cd = fma2(c.Ap, S1, mul2(c.Bp, fma2(a1, b1, mul2(a2, b2))));
    const float2 BA1 = mul2(c.B, a1), BA2 = mul2(c.B, a2), BB1 = mul2(c.B, b1), BB2 = mul2(c.B, b2);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        a.p[q] = fma2(cd, d[q], fma2(BA2, bc2(Gj[q]), fma2(BA1, bc2(Fj[q]), a.p[q])));
        a.p[3 + q] = fma2(BB2, d[q], fma2(c.A, bc2(Gj[q]), a.p[3 + q]));
    }
    a.sG = add2(a.sG, BB1);
    a.sF = add2(a.sF, BB2);
    if constexpr (SYM) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            v[q] = fma2(cd, d[q], fma2(BB1, Gi[q], fma2(BB2, Fi[q], v[q])));
            v[3 + q] = fma2(BA1, d[q], fma2(c.A, Gi[q], v[3 + q]));
        }
        v[6] = add2(v[6], BA1);   // x F_j
        v[7] = add2(v[7], BA2);   // x G_j
    }
}

template <bool ANG, int NT, int NI, int TJ>
constexpr size_t adj_sym_x2_smem_bytes() {
    return (size_t)(ANG ? 4 : 3) * TJ * sizeof(float4) + (size_t)(NT / 32) * adj_comps<ANG>() * TJ * sizeof(float) +
           (size_t)adj_comps<ANG>() * NI * NT * 2 * sizeof(float);
}

template <bool ANG, int NT, int NI, int TJ>
__global__ void __launch_bounds__(NT) adj_sym_x2_kernel(const float4* __restrict__ pos4, const void* __restrict__ Fp,
                                                        const void* __restrict__ Tp, const void* __restrict__ Gp,
                                                        const void* __restrict__ Hp, int f64, SymGeom g,
                                                        RpyConst<float> k, double* __restrict__ partials) {
    static_assert(NI % 2 == 0 && NT >= TJ && TJ % 64 == 0, "packed pairs, one tile load per thread");
    constexpr int NP = NI / 2, C = adj_comps<ANG>(), NV = adj_vals<ANG>(), W = ANG ? 4 : 3;
    extern __shared__ __align__(16) unsigned char adj_sym_smem[];
    float4* s_t = reinterpret_cast<float4*>(adj_sym_smem);    // [w][jj]
    float* s_j = reinterpret_cast<float*>(s_t + W * TJ);      // [warp][c][jj]
    float* s_hi = s_j + (NT / 32) * C * TJ;                   // [c][q][tid]
    float* s_lo = s_hi + C * NI * NT;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float pad = (float)kPadCoord;
    SymItem it;
    if (!sym_item(g, &it)) return;
    const float2 K1 = bc2(k.K1), nK2 = bc2(-k.K2), m3K1 = bc2(-3.f * k.K1), K2x5 = bc2(5.f * k.K2);
    const float2 m1 = bc2(-1.f), m3 = bc2(-3.f), mhalf = bc2(-0.5f), p15 = bc2(1.5f), m75 = bc2(-7.5f);

    auto values = [&](int64_t i, bool in, float away, float* v) {
        const int64_t ii = in ? i : 0;
        if (in) {
            const float4 q = pos4[ii];
            v[0] = q.x; v[1] = q.y; v[2] = q.z;
        } else {
            v[0] = v[1] = v[2] = away;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[3 + c] = in ? load_elem<float>(Fp, f64, 3 * ii + c) : 0.f;
            v[6 + c] = in ? load_elem<float>(Gp, f64, 3 * ii + c) : 0.f;
            v[9 + c] = ANG && in ? load_elem<float>(Tp, f64, 3 * ii + c) : 0.f;
            v[12 + c] = ANG && in ? load_elem<float>(Hp, f64, 3 * ii + c) : 0.f;
        }
        v[15] = 0.f;
    };

    for (int64_t sub = 0; sub < g.m; ++sub) {
        const int64_t b = it.S * g.m + sub;
        const int64_t i0 = b * (int64_t)(NT * NI);
        if (i0 >= g.N) break;
        float2 xi[NP][3], Fi[NP][3], Gi[NP][3], Ti[NP][3], Hi[NP][3];
        Sym6Acc2 a[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float v[2][16];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t i = i0 + (int64_t)(2 * p + h) * NT + tid;
                values(i, i < g.N, -pad, v[h]);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                xi[p][c] = make_float2(v[0][c], v[1][c]);
                Fi[p][c] = make_float2(v[0][3 + c], v[1][3 + c]);
                Gi[p][c] = make_float2(v[0][6 + c], v[1][6 + c]);
                Ti[p][c] = make_float2(v[0][9 + c], v[1][9 + c]);
                Hi[p][c] = make_float2(v[0][12 + c], v[1][12 + c]);
            }
#pragma unroll
            for (int c = 0; c < 9; ++c) a[p].p[c] = bc2(0.f);
            a[p].sG = a[p].sF = a[p].sH = a[p].sT = bc2(0.f);
        }
#pragma unroll
        for (int q = 0; q < NI; ++q) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
                s_hi[(c * NI + q) * NT + tid] = 0.f;
                s_lo[(c * NI + q) * NT + tid] = 0.f;
            }
        }
        const int64_t own = b * g.tb;
        const int64_t ts = it.t0 > own ? it.t0 : own;
        // register prefetch of this thread's j of the next tile
        float nv[16];
        auto fetch = [&](int64_t t) {
            const int64_t j = t * TJ + tid;
            values(j, tid < TJ && t < it.t1 && j < g.N, pad, nv);
        };
        fetch(ts);
        for (int64_t t = ts; t < it.t1; ++t) {
            if (tid < TJ) {
                s_t[tid] = make_float4(-nv[0], -nv[1], -nv[2], nv[3]);
#pragma unroll
                for (int w = 1; w < W; ++w)
                    s_t[w * TJ + tid] = make_float4(nv[4 * w], nv[4 * w + 1], nv[4 * w + 2], nv[4 * w + 3]);
            }
            __syncthreads();
            fetch(t + 1);

            auto step = [&](auto sym_tag, int jj, float2* v) {
                constexpr bool SYM = decltype(sym_tag)::value;
                float jw[4 * W];
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const float4 q = s_t[w * TJ + jj];
                    jw[4 * w] = q.x; jw[4 * w + 1] = q.y; jw[4 * w + 2] = q.z; jw[4 * w + 3] = q.w;
                }
                float2 d[NP][3], r2[NP];
                float mn = 0.f;
#pragma unroll
                for (int p = 0; p < NP; ++p) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) d[p][c] = add2(xi[p][c], bc2(jw[c]));
                    r2[p] = fma2(d[p][0], d[p][0], fma2(d[p][1], d[p][1], mul2(d[p][2], d[p][2])));
                    const float m2 = fminf(r2[p].x, r2[p].y);
                    mn = (p == 0) ? m2 : fminf(mn, m2);
                }
                const bool near = __any_sync(0xffffffffu, mn < k.four_a2);
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    PCoef2 c;
                    float2 gg = bc2(0.f);
                    if (!near) {
                        const float2 invr = make_float2(rsq_far(r2[p].x), rsq_far(r2[p].y));
                        const float2 invr2 = mul2(invr, invr);
                        const float2 invr3 = mul2(invr2, invr);
                        const float2 invr5 = mul2(invr3, invr2);
                        c.A = fma2(K1, invr3, invr);
                        c.B = fma2(nK2, invr5, invr3);
                        c.Ap = mul2(invr3, fma2(m3K1, invr2, m1));   // -1/r^3 - 3 K1/r^5
                        c.Bp = mul2(invr5, fma2(K2x5, invr2, m3));   // -3/r^5 + 5 K2/r^7
                        if constexpr (ANG) {
                            const float2 invr7 = mul2(invr5, invr2);
                            c.g = invr3;
                            c.gp = mul2(m3, invr5);
                            c.ar = mul2(mhalf, invr3);
                            c.arp = mul2(p15, invr5);
                            c.br = c.arp;
                            c.brp = mul2(m75, invr7);
                            gg = c.g;
                        }
                    } else {
                        // exact coefficients of either branch per lane; at r = 0 the
                        // gradient is taken as zero (gg = 0, the derivatives vanish)
                        Coef<float> c0, c1;
                        const bool g0 = exact_coef<float, ANG>(r2[p].x, k, c0);
                        const bool g1 = exact_coef<float, ANG>(r2[p].y, k, c1);
                        c.A = make_float2(c0.A, c1.A);
                        c.B = make_float2(c0.B, c1.B);
                        c.Ap = make_float2(c0.Ap, c1.Ap);
                        c.Bp = make_float2(c0.Bp, c1.Bp);
                        if constexpr (ANG) {
                            c.g = make_float2(c0.g, c1.g);
                            c.gp = make_float2(c0.gp, c1.gp);
                            c.ar = make_float2(c0.ar, c1.ar);
                            c.arp = make_float2(c0.arp, c1.arp);
                            c.br = make_float2(c0.br, c1.br);
                            c.brp = make_float2(c0.brp, c1.brp);
                            gg = make_float2(g0 ? c0.g : 0.f, g1 ? c1.g : 0.f);
                        }
                    }
                    if constexpr (ANG) sym6_pair2<SYM>(d[p], c, gg, Fi[p], Gi[p], Ti[p], Hi[p], jw, a[p], v);
                    else sym3_pair2<SYM>(d[p], c, Fi[p], Gi[p], jw, a[p], v);
                }
            };
            const bool diag = t < own + g.tb;
            float2 v[NV];
            // half tiles: the i-side chains are then as long as the j-side's (64 terms), and the error of
            // both together is below that of whole-tile chains with the j-side added over lanes by a tree
#pragma unroll 1
            for (int j0 = 0; j0 < TJ; j0 += 64) {
                if (diag) {
#pragma unroll 1
                    for (int jj = j0; jj < j0 + 64; ++jj) step(BoolTag<false>{}, jj, v);
                } else {
#pragma unroll 1
                    for (int gr = j0; gr < j0 + 64; gr += 32) {
#pragma unroll
                        for (int c = 0; c < NV; ++c) v[c] = bc2(0.f);
#pragma unroll 1
                        for (int st = 0; st < 32; ++st) {
                            step(BoolTag<true>{}, gr + ((lane + st) & 31), v);
#pragma unroll
                            for (int c = 0; c < NV; ++c) {
                                v[c].x = __shfl_sync(0xffffffffu, v[c].x, (lane + 1) & 31);
                                v[c].y = __shfl_sync(0xffffffffu, v[c].y, (lane + 1) & 31);
                            }
                        }
                        // home again: dX_j -= vector + scalars x (F_j, G_j [, T_j, H_j])
                        float s[NV], jw[4 * W];
#pragma unroll
                        for (int c = 0; c < NV; ++c) s[c] = v[c].x + v[c].y;
#pragma unroll
                        for (int w = 0; w < W; ++w) {
                            const float4 q = s_t[w * TJ + gr + lane];
                            jw[4 * w] = q.x; jw[4 * w + 1] = q.y; jw[4 * w + 2] = q.z; jw[4 * w + 3] = q.w;
                        }
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            float x = fmaf(s[ANG ? 9 : 6], jw[3 + c], fmaf(s[ANG ? 10 : 7], jw[6 + c], s[c]));
                            if constexpr (ANG) x = fmaf(s[11], jw[9 + c], fmaf(s[12], jw[12 + c], x));
                            s_j[(wid * C + c) * TJ + gr + lane] = -x;
                        }
#pragma unroll
                        for (int c = 3; c < C; ++c) s_j[(wid * C + c) * TJ + gr + lane] = s[c];
                    }
                }
                // apply the i-side scalars and fold into the running sums
#pragma unroll
                for (int p = 0; p < NP; ++p) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        float2 x = fma2(a[p].sG, Gi[p][c], fma2(a[p].sF, Fi[p][c], a[p].p[c]));
                        if constexpr (ANG) x = fma2(a[p].sH, Hi[p][c], fma2(a[p].sT, Ti[p][c], x));
                        a[p].p[c] = x;
                    }
                    a[p].sG = a[p].sF = a[p].sH = a[p].sT = bc2(0.f);
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        const int o0 = (c * NI + 2 * p) * NT + tid;
                        fold(&s_hi[o0], &s_lo[o0], a[p].p[c].x);
                        fold(&s_hi[o0 + NT], &s_lo[o0 + NT], a[p].p[c].y);
                    }
                }
            }
            __syncthreads();
            if (!diag) store_j_sums<float, C, NT, TJ>(s_j, g, t, it.S, sub == 0, partials);
        }
        store_i_sums<float, C, NT, NI>(s_hi, s_lo, g, i0, it.S + 1 + it.c, partials);
    }
}

template <typename R, typename K>
cudaError_t launch_form(K kernel, std::atomic<unsigned long long>& attr_devs, size_t dyn, const AdjointArgs& a,
                        const SymGeom& g, dim3 grid, cudaStream_t s) {
    if (cudaError_t e = smem_attr_once(attr_devs, kernel, dyn)) return e;
    kernel<<<grid, a.threads, dyn, s>>>(static_cast<const typename V4<R>::type*>(a.pos4), a.F, a.T, a.G, a.H, a.fp64,
                                        g, make_rpy_const<R>(a.a), a.partials);
    return cudaGetLastError();
}

// Launches the form (occ null) or returns its resident CTAs per SM in *occ.
template <typename R, bool ANG, int NI>
cudaError_t scalar_form(const AdjointArgs* a, const SymGeom& g, dim3 grid, cudaStream_t s, int* occ) {
    constexpr int TJ = sizeof(R) == 8 ? kAdjTileF64 : kAdjTileF32;
    constexpr size_t dyn = adj_sym_s_smem_bytes<R, ANG, 128, NI, TJ>();
    static std::atomic<unsigned long long> attr_devs{0};  // devices whose limit is raised
    if (occ) *occ = sym_occupancy(adj_sym_s_kernel<R, ANG, 128, NI, TJ>, 128, dyn);
    return occ ? cudaSuccess : launch_form<R>(adj_sym_s_kernel<R, ANG, 128, NI, TJ>, attr_devs, dyn, *a, g, grid, s);
}

template <bool ANG, int NT, int NI>
cudaError_t packed_form(const AdjointArgs* a, const SymGeom& g, dim3 grid, cudaStream_t s, int* occ) {
    constexpr int TJ = kAdjTileF32;
    constexpr size_t dyn = adj_sym_x2_smem_bytes<ANG, NT, NI, TJ>();
    static std::atomic<unsigned long long> attr_devs{0};  // devices whose limit is raised
    if (occ) *occ = sym_occupancy(adj_sym_x2_kernel<ANG, NT, NI, TJ>, NT, dyn);
    return occ ? cudaSuccess : launch_form<float>(adj_sym_x2_kernel<ANG, NT, NI, TJ>, attr_devs, dyn, *a, g, grid, s);
}

cudaError_t form(int fp64, int angular, int threads, int ilp, int uj, const AdjointArgs* a, const SymGeom& g, dim3 grid,
                 cudaStream_t s, int* occ) {
    if (fp64)
        return angular ? scalar_form<double, true, 1>(a, g, grid, s, occ) : scalar_form<double, false, 1>(a, g, grid, s, occ);
    if (angular && uj == 3)
        return ilp == 4 ? scalar_form<float, true, 4>(a, g, grid, s, occ) : scalar_form<float, true, 2>(a, g, grid, s, occ);
    if (angular)
        return ilp == 4 ? packed_form<true, 128, 4>(a, g, grid, s, occ) : packed_form<true, 128, 2>(a, g, grid, s, occ);
    if (threads == 256)
        return ilp == 4 ? packed_form<false, 256, 4>(a, g, grid, s, occ) : packed_form<false, 256, 2>(a, g, grid, s, occ);
    return ilp == 4 ? packed_form<false, 128, 4>(a, g, grid, s, occ) : packed_form<false, 128, 2>(a, g, grid, s, occ);
}

}  // namespace

void adjoint_sym_tiling(int fp64, int threads, int ilp, SymPlan* p) {
    p->threads = threads;
    p->ilp = ilp;
    p->tile = fp64 ? kAdjTileF64 : kAdjTileF32;
}

int adjoint_sym_ctas_per_sm(int fp64, int angular, int threads, int ilp, int uj) {
    int n = 0;
    form(fp64, angular, threads, ilp, uj, nullptr, SymGeom{}, dim3(), nullptr, &n);
    return n;
}

cudaError_t launch_adjoint_sym(const AdjointArgs& a, cudaStream_t s) {
    const SymGeom g = sym_geom(a.N, a.sym);
    const dim3 grid = sym_grid(g);
    if (grid.y > 65535 || a.partials == nullptr) return cudaErrorInvalidConfiguration;
    const double c8 = 1.0 / (8.0 * 3.14159265358979323846 * a.eta);
    const cudaError_t err = form(a.fp64, a.angular, a.threads, a.ilp, a.uj, &a, g, grid, s, nullptr);
    count_launches(1);
    if (err != cudaSuccess) return err;
    const SymOut out{{a.dX, a.dF, a.dT}};
    const int C = a.angular ? 9 : 6;
    return a.fp64 ? launch_sym_reduce<double>(a.partials, a.sym, g, C, c8, a.pos4, 0, out, 1, s)
                  : launch_sym_reduce<float>(a.partials, a.sym, g, C, c8, a.pos4, 0, out, 0, s);
}

}  // namespace lmk
