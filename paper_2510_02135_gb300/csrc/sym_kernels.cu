// Symmetric form of the mobility product [u; w] = M(X) [F; T] (Eq.
// block_mobility; NBody solver of Sec. 3.5): every unordered pair is evaluated
// once and applied to both particles.  M is symmetric, so the block that maps
// (F_i, T_i) to particle j is the transpose of the one that maps (F_j, T_j) to
// particle i: separation, reciprocal square root and coefficients are shared.
//
//   pair work (FMA-lane operations per ordered pair)     one-sided  symmetric
//     free space, forces only                                21        15.5
//     free space, all blocks                                 46        41.5
//     single wall, forces only                               80        52
//     single wall, all blocks                               170       134
//
// Schedule:
//   * Item (S, c): the i-blocks of superblock S (m blocks of NT * NI
//     particles) against a chunk of j-tiles of TJ particles, starting at the
//     superblock's own first tile; tiles before a block's own are the business
//     of earlier blocks.
//   * The tiles that hold the block's own particles run one-sided over all
//     ordered pairs (self pairs included), every later tile symmetric.
//   * In a symmetric tile, lane l of a warp meets j = (l + s) mod 32 of a
//     group of 32 in step s.  The j-side sums stay in registers and move one
//     lane per step, so that they are home after 32 steps: one shuffle per
//     value and step, no reduction over lanes and no atomics.
//   * Sums: a thread's i-side per tile in plain FP32, folded into a (hi, lo)
//     pair by TwoSum; the j-side of a warp over 32 * NI particles in FP32, the
//     warps of the CTA added as such a pair.  Both go to FP64 slots that exactly one
//     item writes (j-side slot: its superblock; i-side slots: its chunks), and
//     a second kernel adds a particle's slots in a fixed order: the results
//     are bitwise reproducible.
#include <cuda_runtime.h>

#include <cstdint>

#include "sym_common.cuh"

namespace lmk {
namespace {

// ---------------------------------------------------------------------------
// Scalar form (FP64).  The FP64 pipe takes one warp instruction per 64 cycles
// and SM quarter, so a warp per quarter saturates it and the time is the
// number of FP64 operations: 31 (forces only) or 80 (all blocks) and a
// reciprocal square root per unordered pair.
// ---------------------------------------------------------------------------
template <typename R>
struct PairCoef {
    R A, B, g, ar, br;
};

template <typename R, bool ANG>
__device__ __forceinline__ void far_coef(R r2, const RpyConst<R>& k, PairCoef<R>& o) {
    const R invr = rsq_far(r2);
    const R invr2 = invr * invr;
    const R invr3 = invr2 * invr;
    const R invr5 = invr3 * invr2;
    o.A = fma(k.K1, invr3, invr);
    o.B = fma(-k.K2, invr5, invr3);
    o.g = invr3;
    if constexpr (ANG) {
        o.ar = R(-0.5) * invr3;
        o.br = R(1.5) * invr5;
    }
}

// One side of a pair: p += [M_uF F + M_uT T; M_wF F + M_wT T]; (ex, ey, ez) = g d
// for the target's own d = x_target - x_source.
template <typename R, bool ANG>
__device__ __forceinline__ void apply_side(R dx, R dy, R dz, R ex, R ey, R ez, const PairCoef<R>& o, const R* F,
                                           const R* T, R* p) {
    const R s = o.B * fma(dx, F[0], fma(dy, F[1], dz * F[2]));
    p[0] = fma(s, dx, fma(o.A, F[0], p[0]));
    p[1] = fma(s, dy, fma(o.A, F[1], p[1]));
    p[2] = fma(s, dz, fma(o.A, F[2], p[2]));
    if constexpr (ANG) {
        p[0] = fma(T[1], ez, fma(-T[2], ey, p[0]));
        p[1] = fma(T[2], ex, fma(-T[0], ez, p[1]));
        p[2] = fma(T[0], ey, fma(-T[1], ex, p[2]));
        const R t = o.br * fma(dx, T[0], fma(dy, T[1], dz * T[2]));
        p[3] = fma(F[1], ez, fma(-F[2], ey, fma(t, dx, fma(o.ar, T[0], p[3]))));
        p[4] = fma(F[2], ex, fma(-F[0], ez, fma(t, dy, fma(o.ar, T[1], p[4]))));
        p[5] = fma(F[0], ey, fma(-F[1], ex, fma(t, dz, fma(o.ar, T[2], p[5]))));
    }
}

template <bool ANG, int NT, int NI, int TJ>
__global__ void __launch_bounds__(NT, 4) sym_mdot_f64_kernel(const dvec4* __restrict__ pos4, const void* __restrict__ Fp,
                                                          const void* __restrict__ Tp, int in_f64, SymGeom g,
                                                          RpyConst<double> k, double* __restrict__ partials) {
    constexpr int C = ANG ? 6 : 3;
    constexpr int V = ANG ? 9 : 6;           // values of one j: x, y, z, F, T
    constexpr int NW = NT / 32;
    // lanes that share the rotation over one group of j: with tiles below 32, the 32 / GW parts of a warp meet
    // the same j with different i and are added at the end of the group
    constexpr int GW = TJ < 32 ? TJ : 32;
    __shared__ double s_t[V][TJ];
    __shared__ double s_j[NW][C][TJ];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const double pad = kPadCoord;
    pdl_enter();   // the slot sums may be launched from here on
    SymItem it;
    if (!sym_item(g, &it)) return;
    const int64_t S = it.S, t0 = it.t0, t1 = it.t1;
    const int64_t stride = (int64_t)C * g.N;
    for (int64_t sub = 0; sub < g.m; ++sub) {
        const int64_t b = S * g.m + sub;
        const int64_t i0 = b * (int64_t)(NT * NI);
        if (i0 >= g.N) break;
        double x[NI][3], F[NI][3], Tq[NI][ANG ? 3 : 1], acc[NI][C];
#pragma unroll
        for (int q = 0; q < NI; ++q) {
            const int64_t i = i0 + (int64_t)q * NT + tid;
            const bool in = i < g.N;
            if (in) {
                const dvec4 p = pos4[i];
                x[q][0] = p.x; x[q][1] = p.y; x[q][2] = p.z;
            } else {
                x[q][0] = x[q][1] = x[q][2] = -pad;
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                F[q][c] = in ? load_elem<double>(Fp, in_f64, 3 * i + c) : 0.0;
                if constexpr (ANG) Tq[q][c] = in ? load_elem<double>(Tp, in_f64, 3 * i + c) : 0.0;
            }
#pragma unroll
            for (int c = 0; c < C; ++c) acc[q][c] = 0.0;
        }
        const int64_t own = b * g.tb;
        for (int64_t t = t0 > own ? t0 : own; t < t1; ++t) {
            __syncthreads();   // the previous tile's values and sums are no longer read
            for (int e = tid; e < TJ * V; e += NT) {
                const int v = e / TJ, jj = e % TJ;
                const int64_t j = t * TJ + jj;
                double val;
                if (j < g.N) {
                    if (v < 3) { const dvec4 p = pos4[j]; val = v == 0 ? p.x : (v == 1 ? p.y : p.z); }
                    else val = load_elem<double>(v < 6 ? Fp : Tp, in_f64, 3 * j + (v < 6 ? v - 3 : v - 6));
                } else {
                    val = v < 3 ? pad : 0.0;
                }
                s_t[v][jj] = val;
            }
            __syncthreads();
            const bool diag = t < own + g.tb;
            // "some pair of the warp may overlap" on the high words: an FP64 compare takes the FP64 pipe; the
            // exact form decides for itself
            const int near_hi = __double2hiint(k.four_a2);
            if (diag) {
#pragma unroll 1
                for (int jj = 0; jj < TJ; ++jj) {
                    double Fj[3], Tj[3] = {0.0, 0.0, 0.0};
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        Fj[c] = s_t[3 + c][jj];
                        if constexpr (ANG) Tj[c] = s_t[6 + c][jj];
                    }
#pragma unroll
                    for (int q = 0; q < NI; ++q) {
                        const double dx = x[q][0] - s_t[0][jj], dy = x[q][1] - s_t[1][jj], dz = x[q][2] - s_t[2][jj];
                        const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
                        PairCoef<double> o;
                        if (__any_sync(0xffffffffu, __double2hiint(r2) <= near_hi)) exact_coeffs<double>(r2, k, o.A, o.B, o.g, o.ar, o.br);
                        else far_coef<double, ANG>(r2, k, o);
                        apply_side<double, ANG>(dx, dy, dz, o.g * dx, o.g * dy, o.g * dz, o, Fj, Tj, acc[q]);
                    }
                }
                continue;
            }
#pragma unroll 1
            for (int gr = 0; gr < TJ; gr += GW) {
                double ja[C];
#pragma unroll
                for (int c = 0; c < C; ++c) ja[c] = 0.0;
#pragma unroll 2
                for (int st = 0; st < GW; ++st) {
                    const int jj = gr + ((lane + st) & (GW - 1));
                    double Fj[3], Tj[3] = {0.0, 0.0, 0.0};
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        Fj[c] = s_t[3 + c][jj];
                        if constexpr (ANG) Tj[c] = s_t[6 + c][jj];
                    }
#pragma unroll
                    for (int q = 0; q < NI; ++q) {
                        const double dx = x[q][0] - s_t[0][jj], dy = x[q][1] - s_t[1][jj], dz = x[q][2] - s_t[2][jj];
                        const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
                        PairCoef<double> o;
                        if (__any_sync(0xffffffffu, __double2hiint(r2) <= near_hi)) exact_coeffs<double>(r2, k, o.A, o.B, o.g, o.ar, o.br);
                        else far_coef<double, ANG>(r2, k, o);
                        const double ex = o.g * dx, ey = o.g * dy, ez = o.g * dz;
                        apply_side<double, ANG>(dx, dy, dz, ex, ey, ez, o, Fj, Tj, acc[q]);
                        // the other side: d -> -d leaves the even blocks and negates g d
                        apply_side<double, ANG>(dx, dy, dz, -ex, -ey, -ez, o, F[q], Tq[q], ja);
                    }
#pragma unroll
                    for (int c = 0; c < C; ++c) ja[c] = __shfl_sync(0xffffffffu, ja[c], (lane & ~(GW - 1)) | ((lane + 1) & (GW - 1)));
                }
#pragma unroll
                for (int c = 0; c < C; ++c) {
#pragma unroll
                    for (int o = GW; o < 32; o <<= 1) ja[c] += __shfl_xor_sync(0xffffffffu, ja[c], o);
                    if (lane < GW) s_j[wid][c][gr + lane] = ja[c];
                }
            }
            __syncthreads();
            for (int e = tid; e < TJ * C; e += NT) {
                const int c = e / TJ, jj = e % TJ;
                const int64_t j = t * TJ + jj;
                if (j >= g.N) continue;
                double s = s_j[0][c][jj];
#pragma unroll
                for (int w = 1; w < NW; ++w) s += s_j[w][c][jj];
                const int64_t o = S * stride + (int64_t)c * g.N + j;
                // the superblock's slot of j belongs to this item alone; its blocks add in order
                if (LM_INBOUNDS(o < g.slots * stride, 3, o)) partials[o] = sub == 0 ? s : partials[o] + s;
            }
        }
        const int64_t slot = S + 1 + it.c;
#pragma unroll
        for (int q = 0; q < NI; ++q) {
            const int64_t i = i0 + (int64_t)q * NT + tid;
            if (i >= g.N || !LM_INBOUNDS(slot < g.slots, 3, slot)) continue;
#pragma unroll
            for (int c = 0; c < C; ++c) partials[slot * stride + (int64_t)c * g.N + i] = acc[q][c];
        }
    }
}

// ---------------------------------------------------------------------------
// Packed FP32 form: two i-particles per f32x2 instruction, as the one-sided
// packed kernels; the j-values enter in both lanes as the same scalar and the
// j-side sums are packed too, their two lanes added at the end of a group.
// Tile words: (-x, -y, -z, Fx) (Fy, Fz, Tx | z, Ty) (Tz, z, 0, 0).
// ---------------------------------------------------------------------------
template <bool ANG>
constexpr int sym_words() { return ANG ? 3 : 2; }

template <bool ANG, int NT, int NI, int TJ>
constexpr size_t sym_smem_bytes() {
    return (size_t)sym_words<ANG>() * TJ * sizeof(float4) + running_sum_bytes<float, ANG, NT, NI>() +
           (size_t)(NT / 32) * (ANG ? 6 : 3) * TJ * sizeof(float);
}

struct JVal {
    float2 nx, ny, nz, z;
    float2 F[3], T[3];
};

template <bool ANG, int TJ>
__device__ __forceinline__ JVal sym_load_j(const float4* __restrict__ s_t, int jj) {
    JVal v;
    const float4 w0 = s_t[jj], w1 = s_t[TJ + jj];
    v.nx = bc2(w0.x); v.ny = bc2(w0.y); v.nz = bc2(w0.z);
    v.F[0] = bc2(w0.w); v.F[1] = bc2(w1.x); v.F[2] = bc2(w1.y);
    if constexpr (ANG) {
        const float4 w2 = s_t[2 * TJ + jj];
        v.T[0] = bc2(w1.z); v.T[1] = bc2(w1.w); v.T[2] = bc2(w2.x);
        v.z = bc2(w2.y);
    } else {
        v.z = bc2(w1.z);
        v.T[0] = v.T[1] = v.T[2] = bc2(0.f);
    }
    return v;
}

// Free-space far field of two pairs: acc += (j acts on i), ja += (i acts on j).
template <bool ANG, bool SYM>
__device__ __forceinline__ void sym_far2(float2 dx, float2 dy, float2 dz, float2 r2, float2 K1, float2 nK2,
                                         const JVal& j, const float2* F, const float2* T, float2* acc, float2* ja) {
    const float2 invr = make_float2(rsq_far(r2.x), rsq_far(r2.y));
    const float2 invr2 = mul2(invr, invr);
    const float2 g = mul2(invr2, invr);
    const float2 A = fma2(K1, g, invr);
    const float2 invr5 = mul2(g, invr2);
    const float2 B = fma2(nK2, invr5, g);
    const float2 sj = mul2(B, fma2(dx, j.F[0], fma2(dy, j.F[1], mul2(dz, j.F[2]))));
    acc[0] = fma2(sj, dx, fma2(A, j.F[0], acc[0]));
    acc[1] = fma2(sj, dy, fma2(A, j.F[1], acc[1]));
    acc[2] = fma2(sj, dz, fma2(A, j.F[2], acc[2]));
    if constexpr (SYM) {
        const float2 si = mul2(B, fma2(dx, F[0], fma2(dy, F[1], mul2(dz, F[2]))));
        ja[0] = fma2(si, dx, fma2(A, F[0], ja[0]));
        ja[1] = fma2(si, dy, fma2(A, F[1], ja[1]));
        ja[2] = fma2(si, dz, fma2(A, F[2], ja[2]));
    }
    if constexpr (ANG) {
        const float2 mg = mul2(bc2(-1.f), g);
        const float2 px = mul2(g, dx), py = mul2(g, dy), pz = mul2(g, dz);
        const float2 mx = mul2(mg, dx), my = mul2(mg, dy), mz = mul2(mg, dz);
        const float2 ar = mul2(bc2(-0.5f), g), br = mul2(bc2(1.5f), invr5);
        acc[0] = fma2(j.T[1], pz, fma2(j.T[2], my, acc[0]));
        acc[1] = fma2(j.T[2], px, fma2(j.T[0], mz, acc[1]));
        acc[2] = fma2(j.T[0], py, fma2(j.T[1], mx, acc[2]));
        const float2 tj = mul2(br, fma2(dx, j.T[0], fma2(dy, j.T[1], mul2(dz, j.T[2]))));
        acc[3] = fma2(tj, dx, fma2(ar, j.T[0], fma2(j.F[1], pz, fma2(j.F[2], my, acc[3]))));
        acc[4] = fma2(tj, dy, fma2(ar, j.T[1], fma2(j.F[2], px, fma2(j.F[0], mz, acc[4]))));
        acc[5] = fma2(tj, dz, fma2(ar, j.T[2], fma2(j.F[0], py, fma2(j.F[1], mx, acc[5]))));
        if constexpr (SYM) {
            ja[0] = fma2(T[1], mz, fma2(T[2], py, ja[0]));
            ja[1] = fma2(T[2], mx, fma2(T[0], pz, ja[1]));
            ja[2] = fma2(T[0], my, fma2(T[1], px, ja[2]));
            const float2 ti = mul2(br, fma2(dx, T[0], fma2(dy, T[1], mul2(dz, T[2]))));
            ja[3] = fma2(ti, dx, fma2(ar, T[0], fma2(F[1], mz, fma2(F[2], py, ja[3]))));
            ja[4] = fma2(ti, dy, fma2(ar, T[1], fma2(F[2], mx, fma2(F[0], pz, ja[4]))));
            ja[5] = fma2(ti, dz, fma2(ar, T[2], fma2(F[0], my, fma2(F[1], px, ja[5]))));
        }
    }
}

// The same for two pairs of which some may overlap (either branch, r = 0 too).
template <bool ANG, bool SYM>
__device__ __forceinline__ void sym_exact2(float2 dx, float2 dy, float2 dz, float2 r2, const RpyConst<float>& k,
                                           const JVal& j, const float2* F, const float2* T, float2* acc, float2* ja) {
    constexpr int C = ANG ? 6 : 3;
    const float Fj[3] = {j.F[0].x, j.F[1].x, j.F[2].x}, Tj[3] = {j.T[0].x, j.T[1].x, j.T[2].x};
    float ci[2][C], cj[2][C];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float x = h ? dx.y : dx.x, y = h ? dy.y : dy.x, z = h ? dz.y : dz.x, q = h ? r2.y : r2.x;
        PairCoef<float> o;
        exact_coeffs<float>(q, k, o.A, o.B, o.g, o.ar, o.br);
        const float ex = o.g * x, ey = o.g * y, ez = o.g * z;
#pragma unroll
        for (int c = 0; c < C; ++c) { ci[h][c] = 0.f; cj[h][c] = 0.f; }
        apply_side<float, ANG>(x, y, z, ex, ey, ez, o, Fj, Tj, ci[h]);
        if constexpr (SYM) {
            float Fi[3], Ti[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                Fi[c] = h ? F[c].y : F[c].x;
                if constexpr (ANG) Ti[c] = h ? T[c].y : T[c].x;
            }
            apply_side<float, ANG>(x, y, z, -ex, -ey, -ez, o, Fi, Ti, cj[h]);
        }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
        acc[c] = add2(acc[c], make_float2(ci[0][c], ci[1][c]));
        if constexpr (SYM) ja[c] = add2(ja[c], make_float2(cj[0][c], cj[1][c]));
    }
}

// Wall part (the closed form at the top of wall_kernels.cu) of two pairs, and
// with SYM its transpose for the j-side: the forces' tensor
// A + B e e + C e z + D z e + E z z exchanges C and D, the couplings exchange
// K and L with the sign of the cross products changed, and the torques'
// 3c (e z) and 6c (z e) change places.
template <bool ANG, bool SYM>
__device__ __forceinline__ void sym_wall2(float2 Rx, float2 Ry, float2 zi, float2 a2, const JVal& j, const float2* F,
                                          const float2* T, float2* acc, float2* ja) {
    const float2 Rz = add2(zi, j.z);
    const float2 r2 = fma2(Rx, Rx, fma2(Ry, Ry, mul2(Rz, Rz)));
    const float2 u = make_float2(rsq_far(r2.x), rsq_far(r2.y));
    const float2 ex = mul2(Rx, u), ey = mul2(Ry, u), c = mul2(Rz, u);
    const float2 H = mul2(j.z, u);
    const float2 al = mul2(mul2(a2, u), u);
    const float2 al2 = mul2(al, al);
    const float2 c2 = mul2(c, c), H2 = mul2(H, H), cH = mul2(c, H);
    const float2 alc = mul2(al, c), al2c = mul2(al2, c);
    const float2 A = mul2(u, fma2(al2, fma2(bc2(-10.f / 3.f), c2, bc2(2.f / 3.f)),
                                  fma2(al, fma2(bc2(2.f), c2, bc2(-2.f / 3.f)),
                                       fma2(bc2(2.f), H2, fma2(bc2(-2.f), cH, bc2(-1.f))))));
    const float2 B = mul2(u, fma2(al2, fma2(bc2(70.f / 3.f), c2, bc2(-10.f / 3.f)),
                                  fma2(al, fma2(bc2(-10.f), c2, bc2(2.f)),
                                       fma2(bc2(-6.f), H2, fma2(bc2(6.f), cH, bc2(-1.f))))));
    const float2 Hd = mul2(bc2(2.f), H);
    const float2 Cc = mul2(u, fma2(al2c, fma2(bc2(-140.f / 3.f), c2, bc2(40.f / 3.f)),
                                   fma2(alc, fma2(bc2(20.f), c2, bc2(-4.f)),
                                        fma2(mul2(bc2(12.f), cH), fma2(bc2(-1.f), c, H), Hd))));
    const float2 D = mul2(u, fma2(bc2(-20.f / 3.f), al2c, Hd));
    const float2 E = mul2(u, fma2(al2, fma2(bc2(20.f), c2, bc2(-8.f / 3.f)),
                                  fma2(bc2(-4.f), mul2(al, c2), mul2(bc2(-4.f), H2))));
    const float2 eFj = fma2(ex, j.F[0], fma2(ey, j.F[1], mul2(c, j.F[2])));
    float2 eFi = bc2(0.f);
    {
        const float2 pe = fma2(B, eFj, mul2(Cc, j.F[2]));
        const float2 pz = fma2(D, eFj, fma2(E, j.F[2], acc[2]));
        acc[0] = fma2(A, j.F[0], fma2(pe, ex, acc[0]));
        acc[1] = fma2(A, j.F[1], fma2(pe, ey, acc[1]));
        acc[2] = fma2(A, j.F[2], fma2(pe, c, pz));
    }
    if constexpr (SYM) {
        eFi = fma2(ex, F[0], fma2(ey, F[1], mul2(c, F[2])));
        const float2 pe = fma2(B, eFi, mul2(D, F[2]));
        const float2 pz = fma2(Cc, eFi, fma2(E, F[2], ja[2]));
        ja[0] = fma2(A, F[0], fma2(pe, ex, ja[0]));
        ja[1] = fma2(A, F[1], fma2(pe, ey, ja[1]));
        ja[2] = fma2(A, F[2], fma2(pe, c, pz));
    }
    if constexpr (ANG) {
        const float2 u2 = mul2(u, u);
        const float2 mu2 = mul2(bc2(-1.f), u2);
        const float2 u2d = mul2(bc2(2.f), u2);
        // K1 = -2 (alpha c + H), K2 = 2 (5 alpha c - 3c + 3H), K3 = -2 alpha,
        // L1 = 2 (alpha c - H), L2 = 2 (5 alpha c - 3H), L3 = -2 (10 alpha c^2 - alpha - 6cH), all times u^2
        const float2 px = mul2(u2, ex), py = mul2(u2, ey);
        const float2 mx = mul2(mu2, ex), my = mul2(mu2, ey);
        const float2 pz = mul2(u2, c);
        const float2 mH = mul2(bc2(-1.f), H);
        const float2 hm = add2(alc, mH), hp = add2(alc, H);
        const float2 u2n = mul2(bc2(-1.f), u2d);
        const float2 kz = fma2(u2n, hp, pz), lz = fma2(u2d, hm, pz);     // p_z + K1, p_z + L1
        const float2 mkz = mul2(bc2(-1.f), kz), mlz = mul2(bc2(-1.f), lz);
        const float2 l2c = fma2(bc2(5.f), alc, mul2(bc2(-3.f), H));
        const float2 L2 = mul2(u2d, l2c);
        const float2 K2 = mul2(u2d, fma2(bc2(5.f), alc, fma2(bc2(-3.f), c, mul2(bc2(3.f), H))));
        const float2 K3 = mul2(u2n, al);
        const float2 L3 = mul2(u2n, fma2(bc2(10.f), mul2(al, c2), fma2(bc2(-6.f), cH, mul2(bc2(-1.f), al))));
        const float2 mex = mul2(bc2(-1.f), ex);
        const float2 u3 = mul2(u2, u);
        const float2 Ar = mul2(u3, fma2(bc2(-6.f), c2, bc2(3.5f)));
        const float2 q45 = mul2(bc2(-4.5f), u3), q3 = mul2(bc2(-3.f), u3);
        const float2 c3 = mul2(mul2(bc2(3.f), c), u3), c6 = mul2(mul2(bc2(6.f), c), u3);
        {
            const float2 wT = fma2(ey, j.T[0], mul2(mex, j.T[1]));
            const float2 s = mul2(K2, wT);
            acc[0] = fma2(py, j.T[2], fma2(mkz, j.T[1], fma2(s, ex, acc[0])));
            acc[1] = fma2(kz, j.T[0], fma2(mx, j.T[2], fma2(s, ey, acc[1])));
            acc[2] = fma2(px, j.T[1], fma2(my, j.T[0], fma2(s, c, fma2(K3, wT, acc[2]))));
            const float2 q = fma2(L2, eFj, mul2(L3, j.F[2]));
            const float2 eT = fma2(ex, j.T[0], fma2(ey, j.T[1], mul2(c, j.T[2])));
            const float2 pr = fma2(q45, eT, mul2(c3, j.T[2]));
            acc[3] = fma2(py, j.F[2], fma2(mlz, j.F[1], fma2(q, ey, fma2(Ar, j.T[0], fma2(pr, ex, acc[3])))));
            acc[4] = fma2(lz, j.F[0], fma2(mx, j.F[2], fma2(q, mex, fma2(Ar, j.T[1], fma2(pr, ey, acc[4])))));
            acc[5] = fma2(px, j.F[1], fma2(my, j.F[0],
                          fma2(Ar, j.T[2], fma2(pr, c, fma2(c6, eT, fma2(q3, j.T[2], acc[5]))))));
        }
        if constexpr (SYM) {
            const float2 wT = fma2(ey, T[0], mul2(mex, T[1]));
            const float2 s = mul2(L2, wT);
            ja[0] = fma2(my, T[2], fma2(lz, T[1], fma2(s, ex, ja[0])));
            ja[1] = fma2(mlz, T[0], fma2(px, T[2], fma2(s, ey, ja[1])));
            ja[2] = fma2(mx, T[1], fma2(py, T[0], fma2(s, c, fma2(L3, wT, ja[2]))));
            const float2 q = fma2(K2, eFi, mul2(K3, F[2]));
            const float2 eT = fma2(ex, T[0], fma2(ey, T[1], mul2(c, T[2])));
            const float2 pr = fma2(q45, eT, mul2(c6, T[2]));
            ja[3] = fma2(my, F[2], fma2(kz, F[1], fma2(q, ey, fma2(Ar, T[0], fma2(pr, ex, ja[3])))));
            ja[4] = fma2(mkz, F[0], fma2(px, F[2], fma2(q, mex, fma2(Ar, T[1], fma2(pr, ey, ja[4])))));
            ja[5] = fma2(mx, F[1], fma2(py, F[0],
                         fma2(Ar, T[2], fma2(pr, c, fma2(c3, eT, fma2(q3, T[2], ja[5]))))));
        }
    }
}

template <bool ANG, bool WALL, int NT, int NI, int TJ>
__global__ void __launch_bounds__(NT) sym_mdot_x2_kernel(const float4* __restrict__ pos4, const void* __restrict__ Fp,
                                                         const void* __restrict__ Tp, int in_f64, SymGeom g,
                                                         RpyConst<float> k, float a2s, double* __restrict__ partials) {
    static_assert(NI % 2 == 0 && NT % TJ == 0 && TJ % 32 == 0, "packed pairs, one tile load per thread");
    constexpr int NP = NI / 2, C = ANG ? 6 : 3, W = sym_words<ANG>(), NW = NT / 32;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    float4* s_t = reinterpret_cast<float4*>(dyn_smem);          // [w][jj]
    float* s_hi = reinterpret_cast<float*>(s_t + W * TJ);       // [c][q][tid]
    float* s_lo = s_hi + C * NI * NT;
    float* s_j = s_lo + C * NI * NT;                            // [warp][c][jj]
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float pad = (float)kPadCoord;
    pdl_enter();   // the slot sums may be launched from here on
    SymItem it;
    if (!sym_item(g, &it)) return;
    const int64_t S = it.S, t0 = it.t0, t1 = it.t1;
    const int64_t stride = (int64_t)C * g.N;
    const float2 K1 = bc2(k.K1), nK2 = bc2(-k.K2), a2 = bc2(a2s);

    // register prefetch of this thread's j of the next tile
    float4 np;
    float3 nf, nt;
    auto fetch = [&](int64_t t) {
        const int64_t j = t * TJ + tid;
        if (tid < TJ && t < t1 && j < g.N && LM_INBOUNDS(j >= 0, 1, j)) {
            np = pos4[j];
            const float fj = WALL ? np.w : 1.f;
            nf.x = load_elem<float>(Fp, in_f64, 3 * j + 0);
            nf.y = load_elem<float>(Fp, in_f64, 3 * j + 1);
            nf.z = load_elem<float>(Fp, in_f64, 3 * j + 2);
            if constexpr (WALL) { nf.x *= fj; nf.y *= fj; nf.z *= fj; }
            if constexpr (ANG) {
                nt.x = load_elem<float>(Tp, in_f64, 3 * j + 0);
                nt.y = load_elem<float>(Tp, in_f64, 3 * j + 1);
                nt.z = load_elem<float>(Tp, in_f64, 3 * j + 2);
                if constexpr (WALL) { nt.x *= fj; nt.y *= fj; nt.z *= fj; }
            }
        } else {
            np = make_float4(pad, pad, pad, 0.f);
            nf = make_float3(0.f, 0.f, 0.f);
            nt = make_float3(0.f, 0.f, 0.f);
        }
    };

    for (int64_t sub = 0; sub < g.m; ++sub) {
        const int64_t b = S * g.m + sub;
        const int64_t i0 = b * (int64_t)(NT * NI);
        if (i0 >= g.N) break;
        float2 xi[NP], yi[NP], zi[NP], F[NP][3], T[NP][ANG ? 3 : 1], acc[NP][C];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float v[2][9];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t i = i0 + (int64_t)(2 * p + h) * NT + tid;
                const bool in = i < g.N;
                float f = 1.f;
                if (in) {
                    const float4 q = pos4[i];
                    v[h][0] = q.x; v[h][1] = q.y; v[h][2] = q.z;
                    if constexpr (WALL) f = q.w;
                } else {
                    // far from every particle (above the wall)
                    v[h][0] = -pad; v[h][1] = -pad; v[h][2] = WALL ? pad : -pad;
                }
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    v[h][3 + c] = in ? f * load_elem<float>(Fp, in_f64, 3 * i + c) : 0.f;
                    v[h][6 + c] = ANG && in ? f * load_elem<float>(Tp, in_f64, 3 * i + c) : 0.f;
                }
            }
            xi[p] = make_float2(v[0][0], v[1][0]);
            yi[p] = make_float2(v[0][1], v[1][1]);
            zi[p] = make_float2(v[0][2], v[1][2]);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                F[p][c] = make_float2(v[0][3 + c], v[1][3 + c]);
                if constexpr (ANG) T[p][c] = make_float2(v[0][6 + c], v[1][6 + c]);
            }
#pragma unroll
            for (int c = 0; c < C; ++c) acc[p][c] = bc2(0.f);
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
        const int64_t ts = t0 > own ? t0 : own;
        fetch(ts);
        for (int64_t t = ts; t < t1; ++t) {
            if (tid < TJ) {
                s_t[tid] = make_float4(-np.x, -np.y, -np.z, nf.x);
                if constexpr (ANG) {
                    s_t[TJ + tid] = make_float4(nf.y, nf.z, nt.x, nt.y);
                    s_t[2 * TJ + tid] = make_float4(nt.z, np.z, 0.f, 0.f);
                } else {
                    s_t[TJ + tid] = make_float4(nf.y, nf.z, np.z, 0.f);
                }
            }
            __syncthreads();
            fetch(t + 1);

            // one j (its own per lane when SYM) against the thread's NI particles
            auto step = [&](auto sym_tag, const JVal& j, float2* ja) {
                constexpr bool SYM = decltype(sym_tag)::value;
                float2 dx[NP], dy[NP], dz[NP], r2[NP];
                float mn;
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    dx[p] = add2(xi[p], j.nx);
                    dy[p] = add2(yi[p], j.ny);
                    dz[p] = add2(zi[p], j.nz);
                    r2[p] = fma2(dx[p], dx[p], fma2(dy[p], dy[p], mul2(dz[p], dz[p])));
                    const float m2 = fminf(r2[p].x, r2[p].y);
                    mn = (p == 0) ? m2 : fminf(mn, m2);
                }
                if (__any_sync(0xffffffffu, mn < k.four_a2)) {
                    // the exact form only for the slots with an overlapping (or self) pair in the warp
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        if (__any_sync(0xffffffffu, fminf(r2[p].x, r2[p].y) < k.four_a2))
                            sym_exact2<ANG, SYM>(dx[p], dy[p], dz[p], r2[p], k, j, F[p], T[p], acc[p], ja);
                        else
                            sym_far2<ANG, SYM>(dx[p], dy[p], dz[p], r2[p], K1, nK2, j, F[p], T[p], acc[p], ja);
                    }
                } else {
#pragma unroll
                    for (int p = 0; p < NP; ++p)
                        sym_far2<ANG, SYM>(dx[p], dy[p], dz[p], r2[p], K1, nK2, j, F[p], T[p], acc[p], ja);
                }
                if constexpr (WALL) {
#pragma unroll
                    for (int p = 0; p < NP; ++p)
                        sym_wall2<ANG, SYM>(dx[p], dy[p], zi[p], a2, j, F[p], T[p], acc[p], ja);
                }
            };
            const bool diag = t < own + g.tb;
            if (diag) {
#pragma unroll 1
                for (int jj = 0; jj < TJ; ++jj) step(BoolTag<false>{}, sym_load_j<ANG, TJ>(s_t, jj), nullptr);
            } else {
#pragma unroll 1
                for (int gr = 0; gr < TJ; gr += 32) {
                    float2 ja[C];
#pragma unroll
                    for (int c = 0; c < C; ++c) ja[c] = bc2(0.f);
#pragma unroll (ANG ? 2 : 1)
                    for (int st = 0; st < 32; ++st) {
                        step(BoolTag<true>{}, sym_load_j<ANG, TJ>(s_t, gr + ((lane + st) & 31)), ja);
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            ja[c].x = __shfl_sync(0xffffffffu, ja[c].x, (lane + 1) & 31);
                            ja[c].y = __shfl_sync(0xffffffffu, ja[c].y, (lane + 1) & 31);
                        }
                    }
#pragma unroll
                    for (int c = 0; c < C; ++c) s_j[(wid * C + c) * TJ + gr + lane] = ja[c].x + ja[c].y;
                }
            }
#pragma unroll
            for (int p = 0; p < NP; ++p) {
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const int o0 = (c * NI + 2 * p) * NT + tid;
                    fold(&s_hi[o0], &s_lo[o0], acc[p][c].x);
                    fold(&s_hi[o0 + NT], &s_lo[o0 + NT], acc[p][c].y);
                }
            }
            __syncthreads();
            if (!diag) {
                for (int e = tid; e < TJ * C; e += NT) {
                    const int c = e / TJ, jj = e % TJ;
                    const int64_t j = t * TJ + jj;
                    if (j >= g.N) continue;
                    float hi = s_j[c * TJ + jj], lo = 0.f;
#pragma unroll
                    for (int w = 1; w < NW; ++w) {
                        float x = s_j[(w * C + c) * TJ + jj];
                        fold(&hi, &lo, x);
                    }
                    const double s = (double)hi + (double)lo;   // FP64 operations are dear: two conversions, one add
                    const int64_t o = S * stride + (int64_t)c * g.N + j;
                    // the superblock's slot of j belongs to this item alone; its blocks add in order
                    if (LM_INBOUNDS(o < g.slots * stride, 3, o)) partials[o] = sub == 0 ? s : partials[o] + s;
                }
            }
        }
        const int64_t slot = S + 1 + it.c;
#pragma unroll
        for (int q = 0; q < NI; ++q) {
            const int64_t i = i0 + (int64_t)q * NT + tid;
            if (i >= g.N || !LM_INBOUNDS(slot < g.slots, 3, slot)) continue;
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int o = (c * NI + q) * NT + tid;
                partials[slot * stride + (int64_t)c * g.N + i] = (double)s_hi[o] + (double)s_lo[o];
            }
        }
        __syncthreads();   // the next block reloads the tile
    }
}

constexpr int kSymThreads = 128;
constexpr int kSymWaves = 8;      // items per resident CTA: the largest leave at most an eighth of a wave idle

// A form launches its kernel or, with occ, returns its resident CTAs per SM.
template <bool ANG, int TJ>
cudaError_t f64_form(const MdotArgs* a, const SymGeom& g, dim3 grid, cudaStream_t s, int* occ) {
    if (occ) {
        *occ = sym_occupancy(sym_mdot_f64_kernel<ANG, kSymThreads, 1, TJ>, kSymThreads, 0);
        return cudaSuccess;
    }
    sym_mdot_f64_kernel<ANG, kSymThreads, 1, TJ><<<grid, kSymThreads, 0, s>>>(
        static_cast<const dvec4*>(a->pos4), a->F, ANG ? a->T : nullptr, a->in_f64, g, make_rpy_const<double>(a->a),
        a->partials);
    return cudaGetLastError();
}

template <bool ANG, bool WALL, int NI, int TJ>
cudaError_t x2_form(const MdotArgs* a, const SymGeom& g, dim3 grid, cudaStream_t s, int* occ) {
    constexpr size_t dyn = sym_smem_bytes<ANG, kSymThreads, NI, TJ>();
    if (occ) {
        *occ = sym_occupancy(sym_mdot_x2_kernel<ANG, WALL, kSymThreads, NI, TJ>, kSymThreads, dyn);
        return cudaSuccess;
    }
    static std::atomic<unsigned long long> attr_devs{0};  // devices whose limit is raised
    if (cudaError_t e = smem_attr_once(attr_devs, sym_mdot_x2_kernel<ANG, WALL, kSymThreads, NI, TJ>, dyn)) return e;
    // a plain launch: CTAs that start among the last ones of the kernel before are spread unevenly over the SMs, and
    // a small product lasts as long as its fullest SM (wall, N = 4096: 64 us against 48)
    sym_mdot_x2_kernel<ANG, WALL, kSymThreads, NI, TJ><<<grid, kSymThreads, dyn, s>>>(
        static_cast<const float4*>(a->pos4), a->F, ANG ? a->T : nullptr, a->in_f64, g, make_rpy_const<float>(a->a),
        (float)(a->a * a->a), a->partials);
    return cudaGetLastError();
}

cudaError_t sym_form(int fp64, int angular, int wall, const SymPlan& p, const MdotArgs* a, const SymGeom& g, dim3 grid,
                     cudaStream_t s, int* occ) {
#define LM_FORM64(ANG, TJ) \
    if (fp64 && angular == ANG && p.tile == TJ) return f64_form<ANG, TJ>(a, g, grid, s, occ);
    LM_FORM64(false, 8) LM_FORM64(false, 16) LM_FORM64(false, 32)
    LM_FORM64(true, 8) LM_FORM64(true, 16) LM_FORM64(true, 32)
#undef LM_FORM64
#define LM_FORM(ANG, WALL, NI, TJ) \
    if (!fp64 && angular == ANG && wall == WALL && p.ilp == NI && p.tile == TJ) return x2_form<ANG, WALL, NI, TJ>(a, g, grid, s, occ);
    LM_FORM(false, false, 2, 32) LM_FORM(false, false, 2, 64) LM_FORM(false, false, 4, 128) LM_FORM(false, false, 8, 128)
    LM_FORM(true, false, 2, 32) LM_FORM(true, false, 2, 64) LM_FORM(true, false, 4, 128) LM_FORM(true, false, 8, 128)
    LM_FORM(false, true, 2, 32) LM_FORM(false, true, 2, 64) LM_FORM(false, true, 4, 128)
    LM_FORM(true, true, 2, 32) LM_FORM(true, true, 2, 128)
#undef LM_FORM
    return cudaErrorInvalidConfiguration;
}

}  // namespace

// Products that take the symmetric form.  FP64 with a wall does not (its
// one-sided kernel has no packed form to share the wall part with), nor FP32
// with all blocks in free space from N = 100000 on: 41.5 against 46 operations
// do not pay for the j-side once the one-sided kernel has enough i-blocks for
// eight i-particles per thread and four j per vote (256 x 8).  Device time,
// symmetric / 256 x 8, ms: 40000 2.49 / 2.50, 50000 3.70 / 3.69, 65536 6.32 /
// 6.28, 80000 9.37 / 9.30, 99000 14.23 / 14.15, 131072 24.76 / 23.81, 262144
// 98.6 / 94.6, 524288 394 / 379.  Below the line they are within 1%, and the
// symmetric sums are closer to FP64 (N = 65536: 4.2e-7 / 5.1e-7 of u).
static bool sym_selected(int fp64, int angular, int wall, int64_t N) {
    return wall ? !fp64 : (fp64 || !angular || N < 100000);
}

// i-particles per thread and particles per j-tile.  Small systems are bound by
// the latency of one item, so short tiles and few i-particles make more and
// shorter items; large ones by the FMA pipe, where more i-particles share a
// j-value and its shuffles.  Device time of a product on GB300, us, symmetric at
// (2, 32) / (2, 64) / (4, 128) / (8, 128) and one-sided with its default:
//   forces, free space   N = 100   11 /  13 /  26 /   35 |   21
//                           1000   12 /  15 /  28 /   39 |   22
//                           4096   25 /  23 /  28 /   41 |   32
//                           8192   72 /  61 /  60 /   63 |   78
//                          16384  244 / 206 / 179 /  193 |  255
//                          32768  751 / 720 / 650 /  640 |  845
//                          50021 1686 /1627 /1445 / 1421 | 1916
//   all blocks, free space  1000   14 /  21 /  50 /   59 |   26
//                           4096   51 /  47 /  51 /   82 |   49
//                          10000  217 / 193 / 201 /  201 |  216
//                          16384  482 / 485 / 445 /  454 |  473
//                          32768 1805 /1767 /1667 / 1629 | 1627
//                          65536 7323 /7147 /6643 / 6303 | 6197
//   forces, wall            1000   15 /  21 /  49 |   31     4096   46 /   46 /   49 |   67
//                          16384  495 / 493 / 470 |  719    32768 1882 / 1871 / 1775 | 2600
//   all blocks, wall, (2, 32) / (2, 128)   1000   21 /   59 |   45    4096   99 /  100 |  124
//                                         16384 1203 / 1181 | 1615   32768 4686 / 4604 | 5700
//   FP64 at 8 / 16 / 32 (the FP64 pipe is full at one warp per SM quarter):
//   forces      200   18 /   29 /   52 |  160    1024   50 /   48 /   52 |  151    8001 2138 / 2113 / 2100 | 3390
//   all blocks  200   32 /   56 /  105 |  306    1024  110 /  100 /  105 |  290    8001 4861 / 4811 / 4793 | 7168
static void sym_tiling(int fp64, int angular, int wall, int64_t N, int* ilp, int* tile) {
    *ilp = fp64 ? 1 : 2;
    *tile = !fp64 || N > 3000 ? 32 : (N <= 800 ? 8 : 16);
    if (fp64 || N < (angular && wall ? 5000 : 3500)) return;
    *tile = angular && wall ? 128 : 64;
    if (N < (angular ? 11000 : 10000) || (angular && wall)) return;
    *tile = 128;
    *ilp = wall || N < (angular ? 30000 : 40000) ? 4 : 8;
}

void sym_layout(SymPlan* p, int64_t N, int C, int64_t resident, int64_t chunk) {
    const int64_t block = (int64_t)p->threads * p->ilp;
    const int64_t nblk = (N + block - 1) / block;
    p->tb = block / p->tile;
    p->T = (N + p->tile - 1) / p->tile;
    const int64_t units = nblk * p->T - p->tb * (nblk * (nblk - 1) / 2);
    const int64_t most = std::max<int64_t>(128, ((int64_t)256 << 20) / ((int64_t)C * N * (int64_t)sizeof(double)));
    for (p->m = 1;; p->m *= 2) {
        p->nsuper = (nblk + p->m - 1) / p->m;
        const int64_t want = chunk > 0 ? chunk : std::max<int64_t>(1, units / (kSymWaves * resident * p->m));
        for (p->chunk = want;; p->chunk += want) {
            p->slots = p->nsuper + 1;
            for (int64_t S = 0; S < p->nsuper; ++S)
                p->slots = std::max(p->slots, S + 1 + (p->T - S * p->m * p->tb + p->chunk - 1) / p->chunk);
            if (p->slots <= most) return;
            if (p->chunk > p->m * p->tb) break;
        }
    }
}

bool sym_plan(int fp64, int angular, int wall, int64_t N, int sm_count, SymPlan* p) {
    if (!sym_selected(fp64, angular, wall, N)) return false;
    p->threads = kSymThreads;
    sym_tiling(fp64, angular, wall, N, &p->ilp, &p->tile);
    int occ = 1;
    if (sym_form(fp64, angular, wall, *p, nullptr, SymGeom{}, dim3(), nullptr, &occ) != cudaSuccess) return false;
    sym_layout(p, N, angular ? 6 : 3, (int64_t)std::max(1, occ) * sm_count, 0);
    return true;
}

cudaError_t launch_sym_mdot(const MdotArgs& a, const SymPlan& p, int wall, cudaStream_t s) {
    const SymGeom g = sym_geom(a.N, p);
    const dim3 grid = sym_grid(g);
    if (grid.y > 65535 || a.partials == nullptr) return cudaErrorInvalidConfiguration;
    const double c8 = 1.0 / (8.0 * 3.14159265358979323846 * a.eta);
    if (a.ev_begin) cudaEventRecord(a.ev_begin, s);
    const cudaError_t err = sym_form(a.fp64, a.angular, wall, p, &a, g, grid, s, nullptr);
    if (a.ev_end) cudaEventRecord(a.ev_end, s);
    count_launches(1);
    if (err != cudaSuccess) return err;
    const int C = a.angular ? 6 : 3;
    const SymOut out{{a.lin, a.ang, nullptr}};
    return a.fp64 ? launch_sym_reduce<double>(a.partials, p, g, C, c8, a.pos4, wall, out, a.out_f64, s)
                  : launch_sym_reduce<float>(a.partials, p, g, C, c8, a.pos4, wall, out, a.out_f64, s);
}

}  // namespace lmk
