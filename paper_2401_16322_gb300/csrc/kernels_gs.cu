// Gram-Schmidt of one Arnoldi column in two passes over the basis (FP32, problem sets too large
// for the cooperative column kernel of kernels_mgs.cu).
//
// Modified Gram-Schmidt (Sec. 3.2, the Krylov listing) subtracts one basis vector at a time:
//   h_k = <w - sum_{i<k} h_i v_i, v_k>,   w <- w - h_k v_k,   k = k0 .. j,
// and each step needs the dot of the one before.  In exact arithmetic the same coefficients
// solve a triangular system with the basis's own inner products,
//   (I + L) h = V^T w,   L_{ki} = <v_k, v_i>, i < k
// (the inverse compact WY form of modified Gram-Schmidt: Bjorck, Linear Algebra Appl. 197-198
// (1994); Swirydowicz, Langou, Ananthan, Yang and Thomas, Numer. Linear Algebra Appl. 28 (2021),
// who show that it keeps modified Gram-Schmidt's loss of orthogonality).  L gains one row per
// column, <v_j, v_i>.  So a column takes
//   gs_dots_kernel    reads w = q_{j+1}, q_j and q_{k0} .. q_{j-1} once: <w, q_k> and <q_j, q_k>;
//                     its last block per problem solves the triangular system (FP64), with the
//                     augmented tails, and stores column j of H and row j of L;
//   gs_update_kernel  reads w and q_{k0} .. q_j once: w -= h_k v_k in the order of k, and |w|^2
//                     (the finalisation of the last modified Gram-Schmidt step: h_{j+1,j}, breakdown
//                     test, s_{j+1}, next source scalar).  Not needed after the last column.
//
// Both passes are bound by HBM.  A column reads 2 j + 3 vectors where one pass per step moves 4 j
// (q_{j+1} read and written, v_k and v_{k+1} read at every step), and takes 2 launches where it
// took j + 1.  Each thread holds its 8 vectors of w (and of q_j) in registers
// while the basis streams by.
//
// Sums: the products of four elements are added in FP32 (dot16, as before), and those sums are
// accumulated as unevaluated FP32 pairs (Knuth's TwoSum, 48 bits) instead of in FP64: the FP64
// pipe (2 results per clock and SM) would take 2.7 times the pass's memory time for its two dots
// per element.  The pairs are widened to FP64 before the sums across warps and blocks.
// (Carrying w as such a pair through the update as well made the step 7 % slower and its error
// against FP64 no smaller.)
//
// The dots run over the chunks in descending order and the update in ascending order, so that
// each pass starts on what the one before left in the L2 cache.
// Measured (1001 x 501, 16 shots, Krylov 20): 24.0 -> 12.0 ms a step; error of the step against FP64
// 9.5e-7, as before.
#include <math.h>

#include "ewave_internal.cuh"
#include "flat_vec.cuh"
#include "krylov_finalize.cuh"

namespace ewv {

namespace {

constexpr int GS_VPT = PCHUNK / 4 / NTHREADS;   // 16-byte vectors of a chunk per thread
constexpr int GS_BATCH = NTHREADS / 32 / 2;     // basis vectors per reduction (two sums each, one per warp)
static_assert(GS_VPT * 4 * NTHREADS == PCHUNK, "a chunk is a whole number of vectors per thread");

// The chunk of this block: its problem and 16-byte vectors [q0, q1).
struct Chunk {
    int pid, slot, base, count;
    long long q0;
    int n;                       // vectors in the chunk
    __device__ __forceinline__ Chunk(const ProblemDev* probs, const int* pbase, int nprob, int block) {
        const int2 pc = __ldg(reinterpret_cast<const int2*>(pbase + flat_block_table(nprob)) + block);
        pid = pc.x;
        slot = block;
        base = block - pc.y;
        const ProblemDev* P = probs + pid;
        count = P->pchunks;
        const long long nelem = (long long)P->nfields * P->field_stride;
        const long long e0 = (long long)pc.y * PCHUNK;
        q0 = e0 / 4;
        n = (int)((e0 + PCHUNK < nelem ? (long long)PCHUNK : nelem - e0) / 4);
    }
};

__device__ __forceinline__ void load_chunk(float4 (&v)[GS_VPT], const float4* src, const Chunk& c, int tid) {
    const float4* s = src + c.q0 + tid;
    if (c.n == PCHUNK / 4) {
#pragma unroll
        for (int i = 0; i < GS_VPT; ++i) v[i] = s[i * NTHREADS];
    } else {
#pragma unroll
        for (int i = 0; i < GS_VPT; ++i)
            v[i] = tid + i * NTHREADS < c.n ? s[i * NTHREADS] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

__device__ __forceinline__ void dot_chunk(const float4 (&a)[GS_VPT], const float4 (&b)[GS_VPT], float& hi, float& lo) {
    hi = lo = 0.f;
#pragma unroll
    for (int i = 0; i < GS_VPT; ++i) two_sum_add(hi, lo, dot16(a[i], b[i]));
}

// The sums of a chunk once more, in FP64, where a pair left its range (flat_vec.cuh): a thread per sum.
__device__ __noinline__ void dots_in_fp64(const ProblemDev* P, long long q0, int nv, int j, int k0, double* partials,
                                          size_t stride) {
    auto vec = [&](int k) { return reinterpret_cast<const float4*>(vptr<float>(P, k - 1)) + q0; };   // slot k
    for (int v = threadIdx.x; v < 2 * (j - k0) + 1; v += NTHREADS) {
        const float4* a = vec((v & 1) ? j : j + 1);
        const float4* b = vec(k0 + (v >> 1));
        double s = 0.0;
        for (int q = 0; q < nv; ++q) s += (double)dot16(a[q], b[q]);
        partials[(size_t)v * stride] = s;
    }
}

// One warp: column j of H and row j of L from the totals d[k - k0] = <q_{j+1}, q_k> (k = k0 .. j)
// and l[k - k0] = <q_j, q_k> (k = k0 .. j - 1); tail_{j+1} = J (s_j tail_j) less the h_k v_k tails of
// k = k0 .. j - 1 (the update's finalisation takes k = j).  sh: MAX_M doubles of shared memory.
__device__ void gs_column(const ProblemDev* P, int j, int k0, const double* d, const double* l, double* gram,
                          double* sh, int lane) {
    double* kry = P->kry;
    const int p = P->p;
    const double sj = kry[KRY_S + j];
    const double* tj = kry_tail(kry, j);
    double* tw = kry_tail(kry, j + 1);
    const double w0 = lane < p - 1 ? sj * tj[lane + 1] : 0.0;   // J (s_j tail_j); p <= MAX_P < 32
    double* L = gram + (size_t)(j - 1) * MAX_M;                 // row j
    for (int k = k0; k <= j; ++k) {
        // tail parts of both dots, one warp reduction each
        const double tk = lane < p ? kry_tail(kry, k)[lane] : 0.0;
        double a = w0 * tk, b = (lane < p ? tj[lane] : 0.0) * tk;
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
        }
        if (lane == 0) {
            const double sk = kry[KRY_S + k];
            sh[k - 1] = sk * (d[k - k0] + a);
            if (k < j) L[k - 1] = sj * sk * (l[k - k0] + b);
        }
    }
    __syncwarp();
    // (I + L) h = d by columns: h_k is final once every i < k has been subtracted.  Lane r holds
    // rows k0 + r and k0 + 32 + r (at most MAX_M = 48 of them).
    const int n = j - k0 + 1;
    double h0 = lane < n ? sh[k0 - 1 + lane] : 0.0, h1 = lane + 32 < n ? sh[k0 + 31 + lane] : 0.0;
    const double* g0 = gram + (size_t)(k0 - 1 + lane) * MAX_M + (k0 - 1);
    const double* g1 = g0 + (size_t)32 * MAX_M;
    for (int i = 0; i + 1 < n; ++i) {
        const double hi = __shfl_sync(0xffffffffu, i < 32 ? h0 : h1, i & 31);
        if (lane > i && lane < n) h0 -= g0[i] * hi;
        if (lane + 32 > i && lane + 32 < n) h1 -= g1[i] * hi;
    }
    if (lane < n) {
        kry[KRY_H + (k0 - 1 + lane) * MAX_M + (j - 1)] = h0;
        sh[k0 - 1 + lane] = h0;
    }
    if (lane + 32 < n) {
        kry[KRY_H + (k0 + 31 + lane) * MAX_M + (j - 1)] = h1;
        sh[k0 + 31 + lane] = h1;
    }
    __syncwarp();
    double w = w0;
    if (lane < p) {
        for (int k = k0; k < j; ++k) w -= sh[k - 1] * kry[KRY_S + k] * kry_tail(kry, k)[lane];
        tw[lane] = w;
    }
}

__global__ void __launch_bounds__(NTHREADS, 2)
gs_dots_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ pbase, int nprob, GsArgs ga) {
    __shared__ float2 sred[2 * GS_BATCH][NTHREADS];
    __shared__ double s_tot[2 * MAX_M];
    __shared__ double s_h[MAX_M];
    __shared__ int s_last, s_out;      // s_out: a sum left the range of the pairs
    const Chunk c(probs, pbase, nprob, (int)(gridDim.x - 1 - blockIdx.x));
    const ProblemDev* P = probs + c.pid;
    if (P->kry[KRY_ACTIVE] == 0.0) return;       // Arnoldi stopped
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int j = ga.j, k0 = ga.k0, n = j - k0 + 1;
    float4 w[GS_VPT], p[GS_VPT];
    load_chunk(w, reinterpret_cast<const float4*>(vptr<float>(P, j)), c, tid);          // slot j+1
    load_chunk(p, reinterpret_cast<const float4*>(vptr<float>(P, j - 1)), c, tid);      // slot j
    if (tid == 0) s_out = 0;
    // sums 2 (k - k0) and 2 (k - k0) + 1: <w, q_k> and <q_j, q_k>
    for (int b0 = 0; b0 < n; b0 += GS_BATCH) {
        for (int b = b0; b < n && b < b0 + GS_BATCH; ++b) {
            float dh, dl, lh = 0.f, ll = 0.f;
            if (k0 + b == j) {
                dot_chunk(w, p, dh, dl);
            } else {
                float4 v[GS_VPT];
                load_chunk(v, reinterpret_cast<const float4*>(vptr<float>(P, k0 + b - 1)), c, tid);
                dot_chunk(w, v, dh, dl);
                dot_chunk(p, v, lh, ll);
            }
            sred[2 * (b - b0)][tid] = make_float2(dh, dl);
            sred[2 * (b - b0) + 1][tid] = make_float2(lh, ll);
        }
        __syncthreads();
        if (b0 + warp / 2 < n) {
            float hi = 0.f, lo = 0.f;
#pragma unroll
            for (int i = 0; i < NTHREADS / 32; ++i) {
                const float2 x = sred[warp][lane + 32 * i];
                two_sum_add(hi, lo, x.x);
                lo += x.y;
            }
            double v = (double)hi + (double)lo;
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) {
                ga.partials[(size_t)(2 * b0 + warp) * gridDim.x + c.slot] = v;
                if (out_of_range(v)) s_out = 1;
            }
        }
        __syncthreads();
    }
    if (s_out) {                       // (rare, and the same in every thread)
        dots_in_fp64(P, c.q0, c.n, j, k0, ga.partials + c.slot, gridDim.x);
        __threadfence();
        __syncthreads();
    }
    // the problem's last block sums every total in a fixed order and solves for the column
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(ga.counters + c.pid, 1u) == (unsigned)(c.count - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int v = warp; v < 2 * n; v += NTHREADS / 32) {
        const double* part = ga.partials + (size_t)v * gridDim.x + c.base;
        double s = 0.0;
        for (int t = lane; t < c.count; t += 32) s += __ldcg(part + t);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        // (the sums are kept apart: totals of w first, then of q_j)
        if (lane == 0) s_tot[(v & 1) * MAX_M + (v >> 1)] = s;
    }
    __syncthreads();
    if (warp == 0) {
        double* kry = P->kry;
        bool bad = false;
        for (int v = lane; v < 2 * n; v += 32) bad = bad || !isfinite(s_tot[(v & 1) * MAX_M + (v >> 1)]);
        if (__any_sync(0xffffffffu, bad)) {
            if (lane == 0) {
                kry[KRY_NONFINITE] = 1.0;
                kry[KRY_ACTIVE] = 0.0;
            }
        } else {
            gs_column(P, j, k0, s_tot, s_tot + MAX_M, ga.gram + (size_t)c.pid * MAX_M * MAX_M, s_h, lane);
        }
        if (lane == 0) ga.counters[c.pid] = 0u;
        __threadfence();
    }
}

__global__ void __launch_bounds__(NTHREADS, 3)
gs_update_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ pbase, int nprob, GsArgs ga) {
    __shared__ double red[NTHREADS / 32];
    __shared__ float s_c[MAX_M];
    __shared__ int s_last;
    const Chunk c(probs, pbase, nprob, (int)blockIdx.x);
    const ProblemDev* P = probs + c.pid;
    const double* kry = P->kry;
    if (kry[KRY_ACTIVE] == 0.0) return;
    const int tid = threadIdx.x;
    const int j = ga.j, k0 = ga.k0;
    float4* W = reinterpret_cast<float4*>(vptr<float>(P, j));
    float4 w[GS_VPT];
    load_chunk(w, W, c, tid);
    if (tid <= j - k0) s_c[tid] = (float)(kry[KRY_H + (k0 + tid - 1) * MAX_M + (j - 1)] * kry[KRY_S + k0 + tid]);
    __syncthreads();
    for (int k = k0; k <= j; ++k) {
        float4 v[GS_VPT];
        load_chunk(v, reinterpret_cast<const float4*>(vptr<float>(P, k - 1)), c, tid);
        const float h = s_c[k - k0];
#pragma unroll
        for (int i = 0; i < GS_VPT; ++i) w[i] = axpy16(w[i], h, v[i]);
    }
    DotSum<float4> acc;
#pragma unroll
    for (int i = 0; i < GS_VPT; ++i) {
        if (tid + i * NTHREADS < c.n) W[c.q0 + tid + i * NTHREADS] = w[i];
        acc.add(w[i], w[i]);
    }
    __syncwarp();
    const double bsum = block_total(acc, red, [&](int warp) {
        const float4* wc = reinterpret_cast<const float4*>(vptr<float>(P, j)) + c.q0;
        return warp_dot_in_fp64(wc, wc, c.n, warp);
    });
    StageArgs a{};
    a.fin_mode = FIN_MGS;
    a.fin_j = j;
    a.fin_k = j;
    a.m = ga.m;
    a.tol = ga.tol;
    a.partials = ga.partials;
    a.counters = ga.counters;
    partial_and_finalize_at(P, c.pid, a, bsum, red, &s_last, c.slot, c.base, c.count);
}

}  // namespace

void launch_gs_column(int nchunks, const ProblemDev* probs, const int* pbase, int nprob, const GsArgs& ga,
                      cudaStream_t s) {
    if (nchunks <= 0) return;
    gs_dots_kernel<<<nchunks, NTHREADS, 0, s>>>(probs, pbase, nprob, ga);
    if (ga.j < ga.m) gs_update_kernel<<<nchunks, NTHREADS, 0, s>>>(probs, pbase, nprob, ga);
}

}  // namespace ewv
