// Items, partial-sum slots and their reduction, shared by the symmetric
// product (sym_kernels.cu, which describes the schedule) and the symmetric
// adjoint (adjoint_sym_kernels.cu).
#pragma once

#include <algorithm>

#include "lm_internal.cuh"
#include "pair_common.cuh"
#include "pdl.cuh"

namespace lmk {
namespace {

struct SymGeom {
    int64_t N, T;          // particles, j-tiles
    int64_t m, chunk;      // i-blocks per superblock, j-tiles per item
    int64_t tb;            // j-tiles per i-block
    int64_t slots;         // FP64 slots of every (component, particle)
    int64_t nsuper;        // superblocks
};

template <bool B>
struct BoolTag {
    static constexpr bool value = B;
};

struct SymItem {
    int64_t S, c, t0, t1;  // superblock, chunk, first and end tile
};

__host__ __device__ inline int64_t sym_chunks(const SymGeom& g, int64_t S) {
    return (g.T - S * g.m * g.tb + g.chunk - 1) / g.chunk;
}

// Item of this CTA; false past the end of its grid row.  Row y holds the
// chunks of superblock y, then those of superblock nsuper - 1 - y: a long and
// a short one, so that the rows are alike and hardly any CTA is empty (empty
// CTAs would take a place on an SM while the items are dealt out).
__device__ __forceinline__ bool sym_item(const SymGeom& g, SymItem* it) {
    it->S = blockIdx.y;
    it->c = blockIdx.x;
    const int64_t n = sym_chunks(g, it->S);
    if (it->c >= n) {
        it->c -= n;
        const int64_t S2 = g.nsuper - 1 - it->S;
        if (S2 == it->S || it->c >= sym_chunks(g, S2)) return false;
        it->S = S2;
    }
    it->t0 = it->S * g.m * g.tb + it->c * g.chunk;
    const int64_t e = it->t0 + g.chunk;
    it->t1 = e < g.T ? e : g.T;
    return true;
}

struct SymOut {
    void* o[3];            // components 0..2, 3..5, 6..8; null to skip
};

// out = c8 f_i sum of particle i's slots: j-side slots of the earlier
// superblocks (and of its own, unless it is in the superblock's first block),
// then the i-side slots of its superblock's chunks.  Bound by the latency of
// its loads: the four warps of a CTA take a quarter of the slots of 32 values
// each, eight loads in flight per thread (N = 4096, 33 slots: 14 us with two
// loads in flight and one thread per value).
constexpr int kReduceWarps = 4;

template <typename R>
__global__ void __launch_bounds__(32 * kReduceWarps)
    sym_reduce_kernel(const double* __restrict__ partials, SymGeom g, int64_t block, int C, double c8,
                      const typename V4<R>::type* __restrict__ pos4, int wall, SymOut out, int out_f64) {
    __shared__ double s_p[kReduceWarps][32];
    pdl_enter();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t e = (int64_t)blockIdx.x * 32 + lane;
    const bool in = e < (int64_t)C * g.N;
    const int c = in ? (int)(e / g.N) : 0;
    const int64_t i = in ? e - (int64_t)c * g.N : 0;
    double s = 0.0;
    if (in) {
        const int64_t b = i / block, S = b / g.m;
        const int nj = (int)(S + (b > S * g.m ? 1 : 0));
        const int K = nj + (int)sym_chunks(g, S);
        const int gap = (int)S + 1 - nj;   // slots skipped between the j-side and the i-side
        const double* p = partials + (int64_t)c * g.N + i;
        const int64_t stride = (int64_t)C * g.N;
        const int k1 = K * (wid + 1) / kReduceWarps;
        double t0 = 0.0, t1 = 0.0;
        for (int k = K * wid / kReduceWarps; k < k1; k += 8) {
            double v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = k + q < k1 ? p[(k + q < nj ? k + q : k + q + gap) * stride] : 0.0;
#pragma unroll
            for (int q = 0; q < 8; q += 2) { t0 += v[q]; t1 += v[q + 1]; }
        }
        s = t0 + t1;
    }
    s_p[wid][lane] = s;
    __syncthreads();
    if (wid != 0 || !in) return;
    void* dst = c < 3 ? out.o[0] : (c < 6 ? out.o[1] : out.o[2]);
    if (dst == nullptr) return;
    s = (s + s_p[1][lane]) + (s_p[2][lane] + s_p[3][lane]);
    if (wall) s *= (double)pos4[i].w;
    const int64_t idx = 3 * i + (c % 3);
    if (out_f64) static_cast<double*>(dst)[idx] = c8 * s;
    else static_cast<float*>(dst)[idx] = (float)(c8 * s);
}

inline SymGeom sym_geom(int64_t N, const SymPlan& p) {
    return SymGeom{N, p.T, p.m, p.chunk, p.tb, p.slots, p.nsuper};
}

inline dim3 sym_grid(const SymGeom& g) {
    const int64_t rows = (g.nsuper + 1) / 2;
    int64_t width = 0;
    for (int64_t S = 0; S < rows; ++S) {
        const int64_t S2 = g.nsuper - 1 - S;
        width = std::max(width, sym_chunks(g, S) + (S2 == S ? 0 : sym_chunks(g, S2)));
    }
    return dim3((unsigned)width, (unsigned)rows);
}

// Adds the slots of C components into out (element type out_f64), scaled by
// c8 and, with wall, by the damping factor in pos4.
template <typename R>
cudaError_t launch_sym_reduce(const double* partials, const SymPlan& p, const SymGeom& g, int C, double c8,
                              const void* pos4, int wall, SymOut out, int out_f64, cudaStream_t s) {
    const unsigned blocks = (unsigned)(((int64_t)C * g.N + 31) / 32);
    count_launches(1);
    return launch_pdl(sym_reduce_kernel<R>, dim3(blocks), dim3(32 * kReduceWarps), 0, s, partials, g,
                      (int64_t)p.threads * p.ilp, C, c8, static_cast<const typename V4<R>::type*>(pos4), wall, out,
                      out_f64);
}

template <typename K>
int sym_occupancy(K kernel, int threads, size_t dyn) {
    int n = 0;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, dyn);
    return e == cudaSuccess ? n : 0;
}

}  // namespace
}  // namespace lmk
