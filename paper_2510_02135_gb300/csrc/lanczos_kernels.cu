// FP64 vector kernels of the Krylov (Lanczos) square root, M^{1/2} W
// (libMobility paper, Sec. 3.3): dot products, the three-term update,
// classical Gram-Schmidt against the stored basis (full reorthogonalisation),
// the final combination y = V z and the Philox-4x32-10 normal generator for
// W.  They stream FP64 vectors from HBM; the Gram-Schmidt pair does one FP64
// FMA per 8-byte basis element, so on GB300 (FP64 at 1/64 of the FP32 rate)
// the FP64 pipe, not HBM, bounds it once the basis is long.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>

#include "lm_internal.cuh"
#include "pdl.cuh"
#include "philox.cuh"

namespace lmk {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxBlocks = 1216;   // 8 x 152 SMs: one wave of 256-thread blocks

inline int blocks_for(int64_t n, int per_thread = 4) {
    int64_t b = (n + (int64_t)kThreads * per_thread - 1) / ((int64_t)kThreads * per_thread);
    if (b < 1) b = 1;
    if (b > kMaxBlocks) b = kMaxBlocks;
    return (int)b;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double block_sum(double v) {
    __shared__ double ws[kThreads / 32];
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) ws[wid] = v;
    __syncthreads();
    double t = (threadIdx.x < kThreads / 32) ? ws[threadIdx.x] : 0.0;
    if (wid == 0) t = warp_sum(t);
    __syncthreads();
    return t;  // valid in thread 0
}

__global__ void dot_stage1(const double* __restrict__ x, const double* __restrict__ y, int64_t n,
                           double* __restrict__ red) {
    double acc = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < n; e += (int64_t)gridDim.x * kThreads)
        acc = fma(x[e], y[e], acc);
    acc = block_sum(acc);
    if (threadIdx.x == 0) red[blockIdx.x] = acc;
}

// mode 0: out[0] = sum ; mode 1: out[0] = sqrt(sum), out[1] = sum
__global__ void sum_stage2(const double* __restrict__ red, int nb, double* __restrict__ out, int mode) {
    double acc = 0.0;
    for (int b = threadIdx.x; b < nb; b += kThreads) acc += red[b];
    acc = block_sum(acc);
    if (threadIdx.x == 0) {
        if (mode == 0) out[0] = acc;
        else { out[0] = sqrt(acc); out[1] = acc; }
    }
}

// DGKS test for the second Gram-Schmidt pass: h = [h0, h0^2, h1, h1^2], the
// norms before and after the first pass; the pass runs only if h1 < h0 / sqrt(2).
__device__ __forceinline__ bool second_pass_needed(const double* h) {
    return h == nullptr || h[2] < h[0] * 0.70710678118654752440;
}

// Basis combination for one element e: sum_j c[j] V[j][e], j < m, with c
// staged in shared memory 256 rows at a time.  Eight loads are issued before
// their FMAs and two accumulators alternate, so that a thread keeps eight
// HBM reads and two FP64 FMA chains (64-cycle latency on this GPU) in flight.
__device__ __forceinline__ double basis_combination(const double* __restrict__ V, int m, const double* __restrict__ c,
                                                    int64_t n, int64_t e, double* csh) {
    double a0 = 0.0, a1 = 0.0;
    for (int j0 = 0; j0 < m; j0 += 256) {
        const int mm = (m - j0 < 256) ? (m - j0) : 256;
        __syncthreads();
        if (threadIdx.x < mm) csh[threadIdx.x] = c[j0 + threadIdx.x];
        __syncthreads();
        if (e >= n || !LM_INBOUNDS(j0 + mm <= m, 11, j0 + mm)) continue;
        const double* __restrict__ v = V + (int64_t)j0 * n + e;
        int j = 0;
        for (; j + 8 <= mm; j += 8) {
            double x[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) x[q] = v[(int64_t)(j + q) * n];
#pragma unroll
            for (int q = 0; q < 8; q += 2) {
                a0 = fma(csh[j + q], x[q], a0);
                a1 = fma(csh[j + q + 1], x[q + 1], a1);
            }
        }
        for (; j < mm; ++j) a0 = fma(csh[j], v[(int64_t)j * n], a0);
    }
    return a0 + a1;
}

// y[e] = sum_j z[j] V[j][e] (the Lanczos iterate y = V z).
__global__ void combine_kernel(const double* __restrict__ V, int m, const double* __restrict__ z,
                               double* __restrict__ y, int64_t n) {
    __shared__ double csh[256];
    for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e - threadIdx.x < n;
         e += (int64_t)gridDim.x * kThreads) {
        const double acc = basis_combination(V, m, z, n, e, csh);
        if (e < n) y[e] = acc;
    }
}

__global__ void scale_kernel(const double* __restrict__ x, const double* __restrict__ nrm, double* __restrict__ y,
                             int64_t n) {
    pdl_enter();
    const double inv = 1.0 / nrm[0];
    for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < n; e += (int64_t)gridDim.x * kThreads)
        y[e] = x[e] * inv;
}

__global__ void store_kernel(const double* __restrict__ y, double scale, int64_t N, int angular,
                             void* __restrict__ lin, void* __restrict__ ang, int out_f64) {
    const int64_t n3 = 3 * N;
    const int64_t n = angular ? 2 * n3 : n3;
    for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < n; e += (int64_t)gridDim.x * kThreads) {
        const double v = scale * y[e];
        void* out = (e < n3) ? lin : ang;
        const int64_t idx = (e < n3) ? e : e - n3;
        if (out_f64) static_cast<double*>(out)[idx] = v;
        else static_cast<float*>(out)[idx] = (float)v;
    }
}

__global__ void philox_normals_kernel(uint64_t seed, uint64_t stream, double* __restrict__ W, int64_t n) {
    const int64_t nq = (n + 3) / 4;
    for (int64_t q = (int64_t)blockIdx.x * kThreads + threadIdx.x; q < nq; q += (int64_t)gridDim.x * kThreads) {
        double z[4];
        philox_normals4(seed, stream, (uint64_t)q, z);
#pragma unroll
        for (int t = 0; t < 4; ++t)
            if (4 * q + t < n) W[4 * q + t] = z[t];
    }
}

// Raw Philox-4x32-10 words: out[4 e + t] = word t of philox(ctr[4 e ..], key[2 e ..]).
__global__ void philox_words_kernel(const uint32_t* __restrict__ ctr, const uint32_t* __restrict__ key,
                                    uint32_t* __restrict__ out, int64_t count) {
    for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < count; e += (int64_t)gridDim.x * kThreads) {
        uint32_t c[4] = {ctr[4 * e], ctr[4 * e + 1], ctr[4 * e + 2], ctr[4 * e + 3]};
        philox4x32_10(c, key[2 * e], key[2 * e + 1]);
#pragma unroll
        for (int t = 0; t < 4; ++t) out[4 * e + t] = c[t];
    }
}

// ---------------------------------------------------------------------------
// Single-launch forms: every block writes its partial result, and the last
// block to finish (a device counter, reset by that block) adds the partials
// in block order, so the results are deterministic and equal to the
// two-launch forms'.  They halve the launches of a Lanczos iteration, which
// bound its time at small N.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool last_block_done(unsigned* ctr) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicAdd(ctr, 1u) == gridDim.x - 1);
    __syncthreads();
    return last;
}

// Sum of red[0, nb) in the order of sum_stage2; called by the last block.
__device__ __forceinline__ double final_sum(const double* red, int nb) {
    double acc = 0.0;
    for (int b = threadIdx.x; b < nb; b += kThreads) acc += __ldcg(red + b);
    return block_sum(acc);
}

// mode 0: out[0] = x.y ; mode 1: out[0] = sqrt(x.x), out[1] = x.x
__global__ void dot_fused(const double* __restrict__ x, const double* __restrict__ y, int64_t n, double* red,
                          unsigned* ctr, double* __restrict__ out, int mode) {
    pdl_enter();
    double acc = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < n; e += (int64_t)gridDim.x * kThreads)
        acc = fma(x[e], y[e], acc);
    acc = block_sum(acc);
    if (threadIdx.x == 0) red[blockIdx.x] = acc;
    if (!last_block_done(ctr)) return;
    const double t = final_sum(red, gridDim.x);
    if (threadIdx.x == 0) {
        if (mode == 0) out[0] = t;
        else { out[0] = sqrt(t); out[1] = t; }
        *ctr = 0u;
    }
}

// w -= alpha vk + beta vkm1, then out = (|w|, |w|^2)
__global__ void axpy2_norm_kernel(double* __restrict__ w, const double* __restrict__ vk,
                                  const double* __restrict__ alpha, const double* __restrict__ vkm1,
                                  const double* __restrict__ beta, int64_t n, double* red, unsigned* ctr,
                                  double* __restrict__ out) {
    pdl_enter();
    const double a = alpha[0];
    const double b = (vkm1 != nullptr) ? beta[0] : 0.0;
    double acc = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < n; e += (int64_t)gridDim.x * kThreads) {
        double v = w[e] - a * vk[e];
        if (vkm1 != nullptr) v -= b * vkm1[e];
        w[e] = v;
        acc = fma(v, v, acc);
    }
    acc = block_sum(acc);
    if (threadIdx.x == 0) red[blockIdx.x] = acc;
    if (!last_block_done(ctr)) return;
    const double t = final_sum(red, gridDim.x);
    if (threadIdx.x == 0) { out[0] = sqrt(t); out[1] = t; *ctr = 0u; }
}

// Multi-dot c[j] = v_j . w, j < m.  Block (b, g) takes the rows
// [8g, 8g + 8) over the element chunk [b*kMdChunk, (b+1)*kMdChunk): each
// thread accumulates the eight rows over its kMdElems elements (eight
// independent FP64 chains, w read once per element), the warp reduces the
// eight sums by a transposing butterfly (9 shuffles and adds instead of 40),
// the block adds its four warps and writes red[j * nb + b].  The last block
// of row group g (counter ctr[g]) forms c[j] = sum_b red[j * nb + b] in
// lane-strided order followed by a butterfly, so the result is deterministic.
constexpr int kMdThreads = 128;
constexpr int kMdElems = 8;
constexpr int kMdRows = 8;
constexpr int64_t kMdChunk = (int64_t)kMdThreads * kMdElems;

__global__ void __launch_bounds__(kMdThreads) multidot_rows(const double* __restrict__ V, int m,
                                                            const double* __restrict__ w, int64_t n, double* red,
                                                            unsigned* ctr, double* __restrict__ c,
                                                            const double* __restrict__ cond) {
    pdl_enter();
    if (!second_pass_needed(cond)) return;
    const int nb = gridDim.x, g = blockIdx.y;
    const int j0 = g * kMdRows;
    const int rows = (m - j0 < kMdRows) ? (m - j0) : kMdRows;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t eb = (int64_t)blockIdx.x * kMdChunk + threadIdx.x;
    double acc[kMdRows];
#pragma unroll
    for (int r = 0; r < kMdRows; ++r) acc[r] = 0.0;
#pragma unroll 2
    for (int q = 0; q < kMdElems; ++q) {
        const int64_t e = eb + (int64_t)q * kMdThreads;
        if (e < n) {
            const double we = w[e];
            const double* __restrict__ v = V + (int64_t)j0 * n + e;
#pragma unroll
            for (int r = 0; r < kMdRows; ++r)
                if (r < rows && LM_INBOUNDS(j0 + r < m, 10, j0 + r)) acc[r] = fma(v[(int64_t)r * n], we, acc[r]);
        }
    }
    // transposing butterfly: after the offsets 16, 8 and 4 lane l holds the
    // partial of row l >> 2 (bits 4, 3, 2 of l), completed by offsets 2 and 1
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const bool up = lane & 16;
        const double keep = up ? acc[r + 4] : acc[r], send = up ? acc[r] : acc[r + 4];
        acc[r] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const bool up = lane & 8;
        const double keep = up ? acc[r + 2] : acc[r], send = up ? acc[r] : acc[r + 2];
        acc[r] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    {
        const bool up = lane & 4;
        const double keep = up ? acc[1] : acc[0], send = up ? acc[0] : acc[1];
        acc[0] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
    __shared__ double wsum[kMdThreads / 32][kMdRows];
    if ((lane & 3) == 0) wsum[wid][lane >> 2] = acc[0];
    __syncthreads();
    if (threadIdx.x < rows) {
        double t = wsum[0][threadIdx.x];
#pragma unroll
        for (int q = 1; q < kMdThreads / 32; ++q) t += wsum[q][threadIdx.x];
        red[(int64_t)(j0 + threadIdx.x) * nb + blockIdx.x] = t;
    }
    // the last block of this row group adds the chunks
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicAdd(&ctr[g], 1u) == (unsigned)nb - 1u);
    __syncthreads();
    if (!last) return;
    for (int r = wid; r < rows; r += kMdThreads / 32) {
        const double* pr = red + (int64_t)(j0 + r) * nb;
        double t = 0.0;
        for (int b = lane; b < nb; b += 32) t += __ldcg(pr + b);
        t = warp_sum(t);
        if (lane == 0) c[j0 + r] = t;
    }
    if (threadIdx.x == 0) ctr[g] = 0u;
}

// w -= sum_j c[j] V[j], then out = (|w|, |w|^2).  When the DGKS test skips
// the pass, w is unchanged and its norm is the one the first pass left in
// cond[2], cond[3] (the same kernel over the same w would recompute it bit
// for bit), so one thread copies it.
__global__ void sub_vc_norm_kernel(const double* __restrict__ V, int m, const double* __restrict__ c,
                                   double* __restrict__ w, int64_t n, const double* __restrict__ cond, double* red,
                                   unsigned* ctr, double* __restrict__ out) {
    pdl_enter();
    if (!second_pass_needed(cond)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) { out[0] = cond[2]; out[1] = cond[3]; }
        return;
    }
    __shared__ double csh[256];
    double nrm = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e - threadIdx.x < n;
         e += (int64_t)gridDim.x * kThreads) {
        const double acc = basis_combination(V, m, c, n, e, csh);
        if (e < n) {
            const double v = w[e] - acc;
            w[e] = v;
            nrm = fma(v, v, nrm);
        }
    }
    nrm = block_sum(nrm);
    if (threadIdx.x == 0) red[blockIdx.x] = nrm;
    if (!last_block_done(ctr)) return;
    const double t = final_sum(red, gridDim.x);
    if (threadIdx.x == 0) { out[0] = sqrt(t); out[1] = t; *ctr = 0u; }
}

// ---------------------------------------------------------------------------
// Everything of a Lanczos iteration after its product, in one cooperative
// launch: alpha, the three-term update, the Gram-Schmidt pass (and the second
// one where the DGKS test asks for it), beta and v_{k+1} = w / beta.
//
// For vectors of up to 152 x 512 elements the launches of the separate kernels
// cost more than their work (time per iteration with its product, separate /
// here: N = 300 57 / 36 us, 4096 70 / 49, 16000 238 / 222, FP64 N = 1024 95 /
// 75).  What bounds it is latency: three meetings of about 1 us, and chains of
// FP64 adds of 64 cycles each.  Here CTA b owns the elements
// [b E, (b + 1) E) and keeps its part of w in shared memory; the grid meets
// three times (alpha; norm and dots; norm), and after each meeting every CTA
// adds the CTAs' partial sums itself, all in the same order, so that no
// further meeting distributes the totals and every CTA takes the same branch.
// Dots: a warp takes eight rows at a time (eight FP64 chains, one transposing
// butterfly); the subtraction splits the rows over 256 / E threads per element.
// The CTAs wait for one another, so the launch is cooperative (all resident)
// and every wait has a limit, after which the kernel sets the scalars' error
// word and returns (the host then reports LM_ERR_TIMEOUT).
// ---------------------------------------------------------------------------
constexpr int kStepThreads = 256;
constexpr long long kStepSpinCycles = 4000000000ll;   // about 2 s

struct StepMeet {
    unsigned* ctr;
    unsigned target, arrivals;   // thread 0's: arrivals that end the present meeting, arrivals per meeting
};

__device__ __forceinline__ bool step_meet(StepMeet& meet) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        meet.target += meet.arrivals;
        atomicAdd(meet.ctr, 1u);
        const long long t0 = clock64();
        bool in = true;
        while ((int)(*(volatile unsigned*)meet.ctr - meet.target) < 0) {
            if (clock64() - t0 > kStepSpinCycles) { in = false; break; }
        }
        __threadfence();
        ok = in;
    }
    __syncthreads();
    return ok != 0;
}

// Eight per-lane sums added over the warp: lane l returns the total of value l >> 2.
__device__ __forceinline__ double warp_sum8(double (&v)[8], int lane) {
#pragma unroll
    for (int h = 4, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int r = 0; r < h; ++r) {
            const double keep = up ? v[r + h] : v[r], send = up ? v[r] : v[r + h];
            v[r] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    return v[0];
}

// Sum of this CTA's per-thread values to part[blockIdx.x] (thread 0 writes).
__device__ __forceinline__ void step_put(double v, double* part) {
    v = block_sum(v);
    if (threadIdx.x == 0) part[blockIdx.x] = v;
}

// Sum of the CTAs' values, the same in every CTA; valid in every thread.
__device__ __forceinline__ double step_total(const double* part) {
    __shared__ double tot;
    double v = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += kStepThreads) v += __ldcg(part + b);
    v = block_sum(v);
    if (threadIdx.x == 0) tot = v;
    __syncthreads();
    v = tot;
    __syncthreads();
    return v;
}

// One Gram-Schmidt pass over the rows [0, m): w -= V (V^T w) on this CTA's
// elements.  |w|^2 before the pass is added up as one more row of the dots
// (h0sq), |w|^2 after it by a third meeting (h1sq).  Returns false when a wait
// ran out.
template <int E>
__device__ __forceinline__ bool step_gram_schmidt(const double* __restrict__ V, int m, int64_t n, int64_t e0, double* s_w,
                                                  double* s_c, double* rows, double* norm1, double* h0sq, double* h1sq,
                                                  StepMeet& meet) {
    constexpr int kPer = E / 32;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int G = gridDim.x;
    double we[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) we[q] = s_w[q * 32 + lane];
    for (int j0 = wid * 8; j0 <= m; j0 += kStepThreads / 4) {
        // rows and elements past the end load the last ones (finite, then not used, or times w = 0), so that
        // no branch keeps the loads of two element columns from being in flight together
        const double* __restrict__ row[8];
        double acc[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            row[r] = V + (int64_t)(j0 + r < m ? j0 + r : m - 1) * n;
            acc[r] = 0.0;
        }
#pragma unroll
        for (int q = 0; q < kPer; q += 2) {
            double x[2][8];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t e = e0 + (q + h) * 32 + lane;
                const int64_t ec = e < n ? e : n - 1;
#pragma unroll
                for (int r = 0; r < 8; ++r) x[h][r] = LM_INBOUNDS(ec >= 0, 16, ec) ? row[r][ec] : 0.0;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
#pragma unroll
                for (int r = 0; r < 8; ++r) acc[r] = fma(j0 + r < m ? x[h][r] : we[q + h], we[q + h], acc[r]);
            }
        }
        const double t = warp_sum8(acc, lane);
        if ((lane & 3) == 0 && j0 + (lane >> 2) <= m && LM_INBOUNDS(G <= 152, 17, G))
            rows[(int64_t)(j0 + (lane >> 2)) * G + blockIdx.x] = t;
    }
    if (!step_meet(meet)) return false;
    for (int j0 = wid * 8; j0 <= m; j0 += kStepThreads / 4) {
        double acc[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) acc[r] = 0.0;
#pragma unroll
        for (int q = 0; q < 5; ++q) {   // at most 152 CTAs
            const int b = q * 32 + lane;
            if (q * 32 >= G) break;
            double x[8];
#pragma unroll
            for (int r = 0; r < 8; ++r)
                x[r] = __ldcg(rows + (int64_t)(j0 + r <= m ? j0 + r : m) * G + (b < G ? b : G - 1));
#pragma unroll
            for (int r = 0; r < 8; ++r) acc[r] += b < G ? x[r] : 0.0;
        }
        const double t = warp_sum8(acc, lane);
        if ((lane & 3) == 0 && j0 + (lane >> 2) <= m) s_c[j0 + (lane >> 2)] = t;
    }
    __syncthreads();
    *h0sq = s_c[m];
    // subtraction: kGroups threads share an element's rows (or a thread takes E / 256 elements)
    constexpr int kGroups = E < kStepThreads ? kStepThreads / E : 1;
    constexpr int kElems = E > kStepThreads ? E / kStepThreads : 1;
    __shared__ double s_p[kGroups > 1 ? kStepThreads : 1];
    double v = 0.0;
#pragma unroll
    for (int q = 0; q < kElems; ++q) {
        const int el = (tid % E) + q * kStepThreads, grp = tid / E;
        const int64_t e = e0 + el;
        double a0 = 0.0, a1 = 0.0;
        if (e < n) {
            int j = grp;
            for (; j + kGroups < m; j += 2 * kGroups) {
                a0 = fma(s_c[j], V[(int64_t)j * n + e], a0);
                a1 = fma(s_c[j + kGroups], V[(int64_t)(j + kGroups) * n + e], a1);
            }
            if (j < m) a0 = fma(s_c[j], V[(int64_t)j * n + e], a0);
        }
        double t = a0 + a1;
        if constexpr (kGroups > 1) {
            s_p[tid] = t;
            __syncthreads();
#pragma unroll
            for (int x = 1; x < kGroups; ++x) t += s_p[(tid + x * E) % kStepThreads];
        }
        if (grp == 0) {   // other groups hold the same elements
            t = s_w[el] - t;
            s_w[el] = t;
            v = fma(t, t, v);
        }
    }
    step_put(v, norm1);
    if (!step_meet(meet)) return false;
    *h1sq = step_total(norm1);
    return true;
}

// host_sc: the iteration's scalars [alpha, beta, beta^2, expired wait, -, h0^2,
// -, h1^2] in page-locked host memory (a copy between two iterations would
// hold up the second one's product); sc[1]: beta for the next iteration;
// beta_prev: beta of the iteration before (null at k = 0); part: scratch of
// (5 + 2 m) gridDim.x doubles, m = k + 1; *ctr is a multiple of gridDim.x.
// absent: arrivals that every meeting waits for beyond the grid's (0, but in
// the test of the waits' limit).
template <int E>
__global__ void __launch_bounds__(kStepThreads) lanczos_step_kernel(double* __restrict__ V, int k,
                                                                    const double* __restrict__ w, int64_t n,
                                                                    double* sc, const double* beta_prev,
                                                                    double* part, unsigned* ctr, int always_twice,
                                                                    double* host_sc, int absent) {
    __shared__ double s_w[E];
    extern __shared__ double s_c[];   // k + 1 coefficients, |w|^2
    const int tid = threadIdx.x, G = gridDim.x, m = k + 1;
    const int64_t e0 = (int64_t)blockIdx.x * E;
    const double* vk = V + (int64_t)k * n;
    StepMeet meet{ctr, 0u, (unsigned)(G + absent)};
    if (tid == 0) meet.target = *(volatile unsigned*)ctr / G * G;
    double dot = 0.0;
    for (int q = tid; q < E; q += kStepThreads) {
        const int64_t e = e0 + q;
        const double x = e < n ? w[e] : 0.0;
        s_w[q] = x;
        if (e < n) dot = fma(x, vk[e], dot);
    }
    bool ok = true;
    double alpha = 0.0, h0sq = 0.0, h1sq = 0.0, bsq = 0.0;
    step_put(dot, part);
    ok = step_meet(meet);
    if (ok) {
        alpha = step_total(part);
        const double b = beta_prev != nullptr ? beta_prev[0] : 0.0;
        for (int q = tid; q < E; q += kStepThreads) {
            const int64_t e = e0 + q;
            if (e < n) {
                double x = s_w[q] - alpha * vk[e];
                if (beta_prev != nullptr) x -= b * vk[e - n];
                s_w[q] = x;
            }
        }
        __syncthreads();
        double* rows = part + 3 * (int64_t)G;
        ok = step_gram_schmidt<E>(V, m, n, e0, s_w, s_c, rows, part + G, &h0sq, &h1sq, meet);
        bsq = h1sq;
        double again = 0.0;
        if (ok && (always_twice || h1sq < 0.5 * h0sq))
            ok = step_gram_schmidt<E>(V, m, n, e0, s_w, s_c, rows + (int64_t)(m + 1) * G, part + 2 * G, &again, &bsq,
                                      meet);
    }
    if (!ok) {
        if (tid == 0) host_sc[3] = 1.0;
        return;
    }
    const double inv = rsqrt(bsq), beta = bsq == 0.0 ? 0.0 : bsq * inv;
    for (int q = tid; q < E; q += kStepThreads) {
        const int64_t e = e0 + q;
        if (e < n) V[(int64_t)m * n + e] = s_w[q] * inv;
    }
    if (blockIdx.x == 0 && tid == 0) {
        sc[1] = beta;
        host_sc[0] = alpha; host_sc[1] = beta; host_sc[2] = bsq;
        host_sc[5] = h0sq; host_sc[7] = h1sq;
    }
}

inline int md_blocks(int64_t n) { return (int)((n + kMdChunk - 1) / kMdChunk); }

}  // namespace

size_t lz_red_doubles(int64_t n, int m) {
    const size_t a = (size_t)md_blocks(n) * (size_t)(m < 1 ? 1 : m);
    return a > (size_t)kMaxBlocks ? a : (size_t)kMaxBlocks;
}

size_t lz_ctr_count(int m) { return 1 + (size_t)((m < 1 ? 1 : m) + kMdRows - 1) / kMdRows; }

cudaError_t lz_norm(const double* x, int64_t n, double* red, double* out, cudaStream_t s) {
    const int nb = blocks_for(n);
    dot_stage1<<<nb, kThreads, 0, s>>>(x, x, n, red);
    sum_stage2<<<1, kThreads, 0, s>>>(red, nb, out, 1);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t lz_dot1(const double* x, const double* y, int64_t n, double* red, unsigned* ctr, double* out,
                    int mode, cudaStream_t s) {
    count_launches(1);
    return launch_pdl(dot_fused, dim3(blocks_for(n)), dim3(kThreads), 0, s, x, y, n, red, ctr, out, mode);
}

cudaError_t lz_axpy2_norm(double* w, const double* vk, const double* alpha, const double* vkm1, const double* beta,
                          int64_t n, double* red, unsigned* ctr, double* out, cudaStream_t s) {
    count_launches(1);
    return launch_pdl(axpy2_norm_kernel, dim3(blocks_for(n)), dim3(kThreads), 0, s, w, vk, alpha, vkm1, beta, n, red,
                      ctr, out);
}

cudaError_t lz_multidot1(const double* V, int m, const double* w, int64_t n, double* red, unsigned* ctr, double* c,
                         cudaStream_t s, const double* cond) {
    if (m < 1) return cudaSuccess;
    const int nb = md_blocks(n), ng = (m + kMdRows - 1) / kMdRows;
    if (nb < 1 || ng > 65535) return cudaErrorInvalidConfiguration;
    count_launches(1);
    return launch_pdl(multidot_rows, dim3((unsigned)nb, (unsigned)ng), dim3(kMdThreads), 0, s, V, m, w, n, red, ctr + 1, c,
                      cond);
}

cudaError_t lz_sub_vc_norm(const double* V, int m, const double* c, double* w, int64_t n, double* red,
                           unsigned* ctr, double* out, cudaStream_t s, const double* cond) {
    count_launches(1);
    return launch_pdl(sub_vc_norm_kernel, dim3(blocks_for(n, 1)), dim3(kThreads), 0, s, V, m, c, w, n, cond, red, ctr,
                      out);
}

// Elements per CTA of the one-launch iteration: at most one CTA per SM (152).
static int step_elems(int64_t n) {
    for (int E = 64; E <= 512; E *= 2)
        if (n <= (int64_t)152 * E) return E;
    return 0;
}

size_t lz_step_doubles(int64_t n, int m_max) {
    const int E = step_elems(n);
    if (E == 0 || m_max > 4096) return 0;
    return (size_t)((n + E - 1) / E) * (5 + 2 * (size_t)m_max);
}

cudaError_t lz_step(double* V, int k, const double* w, int64_t n, double* sc, const double* beta_prev, double* part,
                    unsigned* ctr, int always_twice, double* host_sc, cudaStream_t s) {
    const int E = step_elems(n);
    const dim3 grid((unsigned)((n + E - 1) / E));
    const size_t dyn = (size_t)(k + 2) * sizeof(double);
    int absent = 0;
#ifdef LM_DEBUG_BOUNDS
    // tests of the host's side: a refused launch (of every iteration, or from the third on), a wait that runs out
    const char* fault = std::getenv("LM_DEBUG_LANCZOS_STEP");
    if (fault != nullptr && (std::strcmp(fault, "refuse") == 0 || (k >= 2 && std::strcmp(fault, "refuse_later") == 0)))
        return cudaErrorCooperativeLaunchTooLarge;
    absent = fault != nullptr && std::strcmp(fault, "expire") == 0;
#endif
    void* args[] = {&V, &k, &w, &n, &sc, &beta_prev, &part, &ctr, &always_twice, &host_sc, &absent};
    const void* f = E == 64    ? (const void*)lanczos_step_kernel<64>
                    : E == 128 ? (const void*)lanczos_step_kernel<128>
                    : E == 256 ? (const void*)lanczos_step_kernel<256>
                               : (const void*)lanczos_step_kernel<512>;
    const cudaError_t e = cudaLaunchCooperativeKernel(f, grid, dim3(kStepThreads), args, dyn, s);
    if (e == cudaSuccess) count_launches(1);
    return e;
}

cudaError_t lz_scale(const double* x, const double* nrm, double* y, int64_t n, cudaStream_t s) {
    count_launches(1);
    return launch_pdl(scale_kernel, dim3(blocks_for(n)), dim3(kThreads), 0, s, x, nrm, y, n);
}

cudaError_t lz_combine(const double* V, int m, const double* z, double* y, int64_t n, cudaStream_t s) {
    combine_kernel<<<blocks_for(n, 1), kThreads, 0, s>>>(V, m, z, y, n);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t lz_store(const double* y, double scale, int64_t N, int angular, void* lin, void* ang, int out_f64,
                     cudaStream_t s) {
    const int64_t n = (angular ? 6 : 3) * N;
    store_kernel<<<blocks_for(n), kThreads, 0, s>>>(y, scale, N, angular, lin, ang, out_f64);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t lz_philox_normals(uint64_t seed, uint64_t stream, double* W, int64_t n, cudaStream_t s) {
    philox_normals_kernel<<<blocks_for((n + 3) / 4), kThreads, 0, s>>>(seed, stream, W, n);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t lz_philox_words(const uint32_t* ctr, const uint32_t* key, uint32_t* out, int64_t count,
                            cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    philox_words_kernel<<<blocks_for(count), kThreads, 0, s>>>(ctr, key, out, count);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace lmk
