// Small and pointwise kernels around the fused stencil passes:
//  - step clock and per-step source scalars (Ricker derivatives, augmented tail recurrence)
//  - receiver recording (seismogram, Sec. 5.1)
//  - Krylov passes: |x|^2, modified Gram-Schmidt axpy + next dot (Sec. 3.2 listing), the
//    final combination, and the [13/13] Pade exponential of the Hessenberg matrix
//  - Faber coefficients by the trapezoid rule on the unit circle (FP64)
//  - vector copy / swap helpers
#include <math.h>

#include "ewave_internal.cuh"
#include "flat_vec.cuh"
#include "krylov_finalize.cuh"
#include "pdl.cuh"

namespace ewv {

// ---------------------------------------------------------------- clock
__global__ void set_clock_kernel(const ProblemDev* probs, int nprob, double t, double dt) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nprob) return;
    const ProblemDev* P = probs + p;
    P->clk[0] = 0;
    P->tclk[0] = t;
    P->tclk[1] = dt;
    P->kry[KRY_NONFINITE] = 0.0;   // the flag reports non-finite values within one call
}

__global__ void reset_cursor_kernel(const ProblemDev* probs, int nprob) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nprob) return;
    probs[p].clk[1] = 0;
}

// ---------------------------------------------------------------- source scalars
// Ricker r(tau) = (1 - 2 a tau^2) exp(-a tau^2), a = (pi f)^2 (Sec. 4.1).  Its derivatives
// (source_scalars) follow r^(k) = -g^(k+2) / (2a), g = exp(-a tau^2), with the Hermite
// recurrence g^(k) = -2 a tau g^(k-1) - 2 a (k-1) g^(k-2).
__device__ __forceinline__ double ricker(double t, double f, double t0) {
    const double a = (M_PI * f) * (M_PI * f);
    const double tau = t - t0;
    return (1.0 - 2.0 * a * tau * tau) * exp(-a * tau * tau);
}

enum { PRO_FABER = 1, PRO_KRYLOV = 2, PRO_HORK = 3, PRO_RK32 = 4, PRO_RK44 = 5, PRO_LEAPFROG = 6,
       PRO_HORK_HORNER = 7 };

// Source scalars of one step: fills sigma[] (the value added at the source node's v entry in
// each pass) from t_n:
//   Faber: sigma_j = W . y_j, y_0 = e_p, y_1 = F1 y_0, y_2 = F1 y_1 - 2 c1 y_0,
//          y_j = F1 y_{j-1} - c1 y_{j-2}, F1 = (J/dt)/gamma - c0 (tail of Eq. matrix_ampli)
//   HORK:  sigma_i = W . (I + J)^i e_p
//   HORK in Horner form (passes j = m .. 1): sigma_k = W . y_{j+1} with j = m - k,
//          y_{m+1} = e_p, y_j = e_p + (1/j) J y_{j+1}
//   RK3-2 / RK4-4 / leap-frog: f at the stage times
//   Krylov: W stored for the Arnoldi passes
// W[p-1-k] = dt^k r^(k)(t_n) amp / dx^2 (tail scaled by dt).  Warp 0 of the problem's block runs
// the recurrences (lane q holds tail entry q; the shift J is a warp shuffle) and leaves every y
// in shared memory; then one thread per pass forms its W . y.  The chain of one recurrence step
// is a shuffle and one FP64 fma: divisions and the products W . y, each a chain of its own, are
// kept out of it (a launch took 34 us for Horner HORK 20 and 83 us for Faber 60; with the record
// of the step before it in the same launch, Horner 20 on one 601 x 301 shot went from 159 to 131
// us a step).
constexpr int PRO_THREADS = 256;
constexpr int PRO_LD = MAX_P + 1;       // row length of the shared tails (odd: no bank conflicts)

__device__ __forceinline__ void source_scalars(const ProblemDev* P, double tn, double dt, int kind, int m,
                                               double gamma, double c0, double c1, double* sy, double* sw,
                                               double* sr, double* sg) {
    const int tid = threadIdx.x, q = tid & 31;
    if (!P->has_src) return;
    const double scale = P->amp * P->inv_dx2;
    if (kind == PRO_RK32 || kind == PRO_RK44 || kind == PRO_LEAPFROG) {
        // thread 0: f(t_n); 1 and 2: f(t_n + dt/2); 3: f(t_n + dt)
        const int n = kind == PRO_LEAPFROG ? 1 : kind == PRO_RK32 ? 3 : 4;
        if (tid < n) sg[tid] = scale * ricker(tn + (tid == 0 ? 0.0 : tid == 3 ? 1.0 : 0.5) * dt, P->f_peak, P->t0);
        return;
    }
    const int p = P->p;
    const int rows = m < MAX_SIGMA ? m : MAX_SIGMA;
    if (kind == PRO_HORK_HORNER)
        for (int k = tid; k < rows; k += PRO_THREADS) sr[k] = 1.0 / (double)(m - k);
    __syncthreads();
    if (tid < 32) {
        // W_q = dt^k r^(k)(t_n) scale with k = p-1-q: every lane runs the Hermite recurrence
        // g^(k) = -2 a tau g^(k-1) - 2 a (k-1) g^(k-2) and keeps its own term
        const int kq = p - 1 - q;
        const double a = (M_PI * P->f_peak) * (M_PI * P->f_peak);
        const double tau = tn - P->t0;
        double gm2 = exp(-a * tau * tau), gm1 = -2.0 * a * tau * gm2, gk = 0.0, dk = 1.0, pw = 1.0;
        for (int k = 2; k < p + 2; ++k) {
            const double g = -2.0 * a * tau * gm1 - 2.0 * a * (double)(k - 1) * gm2;
            if (k - 2 == kq) {
                gk = g;
                dk = pw;
            }
            pw *= dt;
            gm2 = gm1;
            gm1 = g;
        }
        const double W = (q < p) ? dk * (-gk / (2.0 * a)) * scale : 0.0;
        if (q < MAX_P) sw[q] = W;
        if (kind != PRO_KRYLOV) {
            const bool up_in = q + 1 < p;
            const double e = (q == p - 1) ? 1.0 : 0.0;
            auto shift = [&](double y) {           // J y
                const double u = __shfl_down_sync(0xffffffffu, y, 1);
                return up_in ? u : 0.0;
            };
            double y = e;
            if (kind == PRO_FABER) {
                const double ig = 1.0 / gamma / dt;
                double ym = 0.0;
                for (int j = 0; j < rows; ++j) {
                    if (q < p) sy[j * PRO_LD + q] = y;
                    const double cj = (j == 1) ? 2.0 * c1 : c1;       // (y_{-1} = 0)
                    const double t = -c0 * y - cj * ym;
                    ym = y;
                    y = fma(ig, shift(y), t);
                }
            } else if (kind == PRO_HORK_HORNER) {
                for (int k = 0; k < rows; ++k) {
                    if (q < p) sy[k * PRO_LD + q] = y;
                    y = fma(shift(y), sr[k], e);
                }
            } else {
                for (int i = 0; i < rows; ++i) {                       // y_i = (I + J) y_{i-1}
                    if (q < p) sy[i * PRO_LD + q] = y;
                    y = y + shift(y);
                }
            }
        }
    }
    __syncthreads();
    if (kind == PRO_KRYLOV) return;
    for (int k = tid; k < rows; k += PRO_THREADS) {
        double s0 = 0.0, s1 = 0.0;
        for (int e = 0; e < p; e += 2) {
            s0 = fma(sw[e], sy[k * PRO_LD + e], s0);
            if (e + 1 < p) s1 = fma(sw[e + 1], sy[k * PRO_LD + e + 1], s1);
        }
        sg[k] = s0 + s1;
    }
}

// Stores what source_scalars left in shared memory.
__device__ __forceinline__ void publish_scalars(const ProblemDev* P, int kind, int m, const double* sw,
                                                const double* sg) {
    const int tid = threadIdx.x;
    if (!P->has_src) {
        for (int s = tid; s < MAX_SIGMA; s += PRO_THREADS) P->sigma[s] = 0.0;
        if (kind == PRO_KRYLOV && tid < MAX_P) P->kry[KRY_W + tid] = 0.0;
        return;
    }
    if (kind == PRO_KRYLOV) {
        if (tid < MAX_P) P->kry[KRY_W + tid] = sw[tid];
        return;
    }
    const int n = kind == PRO_LEAPFROG ? 1 : kind == PRO_RK32 ? 3 : kind == PRO_RK44 ? 4 : m < MAX_SIGMA ? m : MAX_SIGMA;
    for (int k = tid; k < n; k += PRO_THREADS) P->sigma[k] = sg[k];
}

// ---------------------------------------------------------------- between two steps
// One block per problem: records sample clk[1] from vector `vec` (record), advances the clock
// and prepares the source scalars of the step that follows (kind >= 0); or, before the first
// step of a call, only the latter.  One launch between two steps instead of two: at the sizes
// where a pass takes a few microseconds every launch counts.
template <typename T>
__global__ void __launch_bounds__(PRO_THREADS)
between_kernel(const ProblemDev* probs, int nprob, int record, int vec, int kind, int m, double gamma, double c0,
               double c1) {
    __shared__ double sy[MAX_SIGMA * PRO_LD];
    __shared__ double sw[MAX_P];
    __shared__ double sr[MAX_SIGMA];
    __shared__ double sg[MAX_SIGMA];
    __shared__ long long s_clk;
    __shared__ double s_t[2];
    const ProblemDev* P = probs + blockIdx.x;
    pdl_trigger();
    if (kind >= 0) {
        // the scalars hang on the clock alone, which stands still during a step: they are formed
        // before the wait for the step's last pass, with the clock as it is now (checked below).
        // Leap-frog, 16 steps of 16 shots on 1001 x 501: 1266 -> 1230 us.
        if (threadIdx.x == 0) {
            s_clk = *(volatile const long long*)P->clk;
            s_t[0] = ((volatile const double*)P->tclk)[0];
            s_t[1] = ((volatile const double*)P->tclk)[1];
        }
        __syncthreads();
        source_scalars(P, s_t[0] + (double)(s_clk + (record ? 1 : 0)) * s_t[1], s_t[1], kind, m, gamma, c0, c1, sy, sw,
                       sr, sg);
        __syncthreads();
    }
    pdl_wait();
    const long long clk = *(volatile const long long*)P->clk, step = clk + (record ? 1 : 0);
    const double t0 = ((volatile const double*)P->tclk)[0], dt = ((volatile const double*)P->tclk)[1];
    if (record) {
        const long long cur = P->clk[1];
        if (P->seismo && cur < P->capacity) {
            const T* u = vptr<T>(P, vec);
            T* out = (T*)P->seismo + cur * P->rec_stride;
            for (int r = PRO_THREADS - 1 - (int)threadIdx.x; r < P->nrec; r += PRO_THREADS) out[r] = u[P->rec_off[r]];
        }
        __syncthreads();          // every thread has read the clock
        if (threadIdx.x == 0) {
            P->clk[1] = cur + 1;
            P->clk[0] = step;
        }
    }
    if (kind >= 0) {
        if (clk != s_clk || t0 != s_t[0] || dt != s_t[1]) {      // (the same in every thread)
            __syncthreads();
            source_scalars(P, t0 + (double)step * dt, dt, kind, m, gamma, c0, c1, sy, sw, sr, sg);
            __syncthreads();
        }
        publish_scalars(P, kind, m, sw, sg);
    }
}

// ---------------------------------------------------------------- adjoint source
// lambda_u[rec] += values[shot][rec] (the transpose of recording, R^T r); one block per shot, one
// thread per receiver.  Of coincident receivers the first adds all their values in order, so the
// sums are deterministic (62 us with one thread per shot adding 200 receivers one after another).
// link[r] leads from a receiver to the next on its node (0: none), complemented where r is not the
// first there: the list is made with the receivers, because a search among them here would grow
// with their square (2 shots of 32768: 85 ms with the search, 0.15 ms with the links; 2 of 4096: 1.4
// and 0.02 ms).
template <typename T>
__global__ void inject_kernel(T* adj, long long vec_elems, const T* values, const int* rec, const int* nrec,
                              int max_rec) {
    const int sh = blockIdx.x;
    T* lam = adj + (long long)sh * vec_elems;
    const T* val = values + (long long)sh * max_rec;
    const int n = nrec[sh];
    const int* off = rec + (long long)sh * 2 * max_rec;
    const int* link = off + n;
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
        int e = link[r];
        if (e < 0) continue;
        T v = lam[off[r]] + val[r];
        for (; e > 0; e = ~link[e]) v += val[e];
        lam[off[r]] = v;
    }
}

// out[o] = sum_s in[s][o], shots summed in index order (deterministic).
template <typename T>
__global__ void sum_shots_kernel(const T* in, T* out, long long n, int nshots) {
    for (long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x; o < n;
         o += (long long)gridDim.x * blockDim.x) {
        T acc = T(0);
        for (int s = 0; s < nshots; ++s) acc += in[(long long)s * n + o];
        out[o] = acc;
    }
}

// ---------------------------------------------------------------- pointwise Krylov passes
// Each uses the stencil kernels' tile decomposition so that partial index == block index.

template <typename T>
__global__ void __launch_bounds__(NTHREADS)
point_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ tile_prob,
             PointArgs pa) {
    __shared__ double red[NTHREADS / 32];
    __shared__ int s_last;
    const int pid = tile_prob[blockIdx.x];
    const ProblemDev* P = probs + pid;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int nx = P->nx, ny = P->ny, pitch = P->pitch;
    const int lt = blockIdx.x - P->tile_base;
    // tile (x, y[, z chunk of KC3 planes]); 2D problems have nz = 1 and one z tile
    const int nz = P->nz > 1 ? P->nz : 1;
    const int nf = P->nfields;   // 4 (2D) or 6 (3D: w_z and psi added)
    const int rr = lt / P->tiles_x;
    const int x0 = (lt % P->tiles_x) * BX, y0 = (rr % P->tiles_y) * BY;
    const int k0 = nz > 1 ? (rr / P->tiles_y) * KC3 : 0;
    const int k1 = nz > 1 ? min(k0 + KC3, nz) : 1;
    const long long ps = (long long)ny * pitch;
    const long long fstr = P->field_stride;
    double* kry = P->kry;

    if (pa.mode == 1 && kry[KRY_ACTIVE] == 0.0) return;
    if (pa.mode == 3 || pa.mode == 4 || pa.mode == 6) {
        T* S = vptr<T>(P, pa.mode == 6 ? pa.dst : pa.src);
        T* Dd = vptr<T>(P, pa.dst);
        for (int kz = k0; kz < k1; ++kz)
        for (int b = 0; b < VY; ++b)
            for (int c = 0; c < VX; ++c) {
                const int i = x0 + tx + c * TPX, j = y0 + ty + b * TPY;
                if (i >= nx || j >= ny) continue;
                const long long o = kz * ps + (long long)j * pitch + i;
                for (int f = 0; f < nf; ++f) {
                    if (!((pa.fmask >> f) & 1)) continue;
                    if (pa.mode == 6) {
                        Dd[f * fstr + o] = T(0);
                        continue;
                    }
                    const T s = S[f * fstr + o];
                    if (pa.mode == 4) S[f * fstr + o] = Dd[f * fstr + o];
                    Dd[f * fstr + o] = s;
                }
            }
        return;
    }
    if (pa.mode == 2) {
        // u^{n+1} = beta sum_{k=1}^{meff} e_k s_k q_k  (q_1 is the state itself)
        if (kry[KRY_NONFINITE] != 0.0) return;
        const int meff = (int)kry[KRY_MEFF];
        const double beta = kry[KRY_BETA];
        T coef[MAX_M];
        for (int k = 1; k <= meff; ++k) coef[k - 1] = (T)(beta * kry[KRY_E + k - 1] * kry[KRY_S + k]);
        T* St = vptr<T>(P, 0);
        for (int kz = k0; kz < k1; ++kz)
        for (int b = 0; b < VY; ++b)
            for (int c = 0; c < VX; ++c) {
                const int i = x0 + tx + c * TPX, j = y0 + ty + b * TPY;
                if (i >= nx || j >= ny) continue;
                const long long o = kz * ps + (long long)j * pitch + i;
                for (int f = 0; f < nf; ++f) {
                    T acc = T(0);
                    for (int k = 1; k <= meff; ++k) acc += coef[k - 1] * vptr<T>(P, k - 1)[f * fstr + o];
                    St[f * fstr + o] = acc;
                }
            }
        return;
    }
    // mode 0 (norm of the state) or 1 (MGS pass k of Arnoldi step j):
    // q_{j+1} -= h_{k,j} s_k q_k, then partial <q_{j+1}, q_{k+1}> (k < j) or |q_{j+1}|^2.
    float accf = 0.f;
    double accd = 0.0;
    T* W = nullptr;
    const T* Qk = nullptr;
    const T* Qn = nullptr;
    T coef = T(0);
    if (pa.mode == 0) {
        Qn = vptr<T>(P, 0);
    } else {
        W = vptr<T>(P, pa.j);                  // slot j+1
        Qk = vptr<T>(P, pa.k - 1);             // slot k
        coef = (T)(kry[KRY_H + (pa.k - 1) * MAX_M + (pa.j - 1)] * kry[KRY_S + pa.k]);
        Qn = pa.k < pa.j ? vptr<T>(P, pa.k) : nullptr;   // slot k+1 (or w itself)
    }
    for (int kz = k0; kz < k1; ++kz)
    for (int b = 0; b < VY; ++b)
        for (int c = 0; c < VX; ++c) {
            const int i = x0 + tx + c * TPX, j = y0 + ty + b * TPY;
            if (i >= nx || j >= ny) continue;
            const long long o = kz * ps + (long long)j * pitch + i;
            for (int f = 0; f < nf; ++f) {
                if ((f == 2 && i >= nx - 1) || (f == 3 && j >= ny - 1) || (f == 4 && kz >= nz - 1))
                    continue;
                T val;
                T other;
                if (pa.mode == 0) {
                    val = Qn[f * fstr + o];
                    other = val;
                } else {
                    val = W[f * fstr + o] - coef * Qk[f * fstr + o];
                    W[f * fstr + o] = val;
                    other = Qn ? Qn[f * fstr + o] : val;
                }
                if (sizeof(T) == 4) accf = fmaf((float)val, (float)other, accf);
                else accd = fma((double)val, (double)other, accd);
            }
        }
    if (pa.mode == 1 && pa.k == pa.j && pa.j == pa.m) return;   // h_{m+1,m} unused
    const double bsum = block_sum_fixed((double)accf + accd, red);
    StageArgs a{};
    a.fin_mode = pa.mode == 0 ? FIN_NORM0 : FIN_MGS;
    a.fin_j = pa.j;
    a.fin_k = pa.k;
    a.m = pa.m;
    a.tol = pa.tol;
    a.partials = pa.partials;
    a.counters = pa.counters;
    partial_and_finalize(P, pid, a, bsum, red, &s_last);
}

// ---------------------------------------------------------------- flat pointwise passes
// Modes 0 (|q_1|^2), 1 (MGS pass) and 2 (Krylov combine) over whole padded vectors: every
// pad element is zero in every vector, so the flat sums and updates equal the masked ones.
// Block b handles elements [c PCHUNK, (c + 1) PCHUNK) of problem p ((p, c) from the block
// table after the prefix sums), with
// 16-byte vector loads; its partial dot product goes to slot b, and the problem's last block
// sums the partials in a fixed order (deterministic, no waiting).
__device__ __forceinline__ int flat_problem(const int* __restrict__ base, int nprob, int b) {
    int lo = 0, hi = nprob - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(base + mid) <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <typename T>
__global__ void __launch_bounds__(NTHREADS)
point_flat_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ pbase, int nprob,
                  PointArgs pa) {
    using V = typename Vec16<T>::type;
    constexpr int NV = Vec16<T>::N;
    __shared__ double red[NTHREADS / 32];
    __shared__ int s_last;
    __shared__ T s_coef[MAX_M];
    const int2 pc = __ldg(reinterpret_cast<const int2*>(pbase + flat_block_table(nprob)) + blockIdx.x);
    const int pid = pc.x;
    const ProblemDev* P = probs + pid;
    double* kry = P->kry;
    if ((pa.mode == 1 || pa.mode == 5) && kry[KRY_ACTIVE] == 0.0) return;
    if (pa.mode == 2 && (kry[KRY_NONFINITE] != 0.0 || kry[KRY_SKIP] != 0.0)) return;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int nf = P->nfields;   // 4 (2D) or 6 (3D: w_z and psi added)
    const long long nelem = (long long)nf * P->field_stride;
    const long long e0 = (long long)pc.y * PCHUNK;
    const long long e1 = e0 + PCHUNK < nelem ? e0 + PCHUNK : nelem;
    const long long q0 = e0 / NV, q1 = e1 / NV;
    if (pa.mode == 2) {
        // u^{n+1} = beta sum_{k=1}^{meff} e_k s_k q_k  (q_1 is the state itself)
        const int meff = (int)kry[KRY_MEFF];
        const double beta = kry[KRY_BETA];
        for (int k = tid; k < meff; k += NTHREADS) s_coef[k] = (T)(beta * kry[KRY_E + k] * kry[KRY_S + k + 1]);
        __syncthreads();
        V* St = pa.out ? reinterpret_cast<V*>(static_cast<T*>(pa.out) + (long long)pid * pa.out_stride)
                       : reinterpret_cast<V*>(vptr<T>(P, pa.dst));
        // eight vectors a thread at a time: eight loads in flight for every basis vector
        constexpr int G = 8;
        for (long long q = q0 + tid; q < q1; q += G * NTHREADS) {
            V acc[G];
#pragma unroll
            for (int g = 0; g < G; ++g) acc[g] = V{};
            for (int k = 1; k <= meff; ++k) {
                const V* B = reinterpret_cast<const V*>(vptr<T>(P, k - 1));
#pragma unroll
                for (int g = 0; g < G; ++g)
                    if (q + g * NTHREADS < q1) fma16(acc[g], s_coef[k - 1], B[q + g * NTHREADS]);
            }
#pragma unroll
            for (int g = 0; g < G; ++g)
                if (q + g * NTHREADS < q1) St[q + g * NTHREADS] = acc[g];
        }
        return;
    }
    DotSum<V> acc;
    if (pa.mode == 0) {
        const V* Q = reinterpret_cast<const V*>(vptr<T>(P, 0));
        for (long long q = q0 + tid; q < q1; q += NTHREADS) {
            const V a = Q[q];
            acc.add(a, a);
        }
    } else if (pa.mode == 7) {
        const V* W = reinterpret_cast<const V*>(vptr<T>(P, pa.j));      // slot j+1
        for (long long q = q0 + tid; q < q1; q += NTHREADS) {
            const V w = W[q];
            acc.add(w, w);
        }
    } else if (pa.mode == 5) {
        // <q_{j+1}, q_k> after the matrix-vector product (its finalisation is FIN_MATVEC)
        const V* W = reinterpret_cast<const V*>(vptr<T>(P, pa.j));      // slot j+1
        const V* D = reinterpret_cast<const V*>(vptr<T>(P, pa.k - 1));  // slot k
        for (long long q = q0 + tid; q < q1; q += NTHREADS) acc.add(W[q], D[q]);
    } else {
        V* W = reinterpret_cast<V*>(vptr<T>(P, pa.j));                  // slot j+1
        const V* Qk = reinterpret_cast<const V*>(vptr<T>(P, pa.k - 1));   // slot k
        const V* Qn = pa.k < pa.j ? reinterpret_cast<const V*>(vptr<T>(P, pa.k)) : nullptr;
        const T coef = (T)(kry[KRY_H + (pa.k - 1) * MAX_M + (pa.j - 1)] * kry[KRY_S + pa.k]);
#pragma unroll 2
        for (long long q = q0 + tid; q < q1; q += NTHREADS) {
            const V wq = W[q], qk = Qk[q];
            // every operand is loaded before the store: the loads may not move past a store
            // the compiler cannot prove disjoint, which would cost a second memory round trip
            const V qn = Qn ? Qn[q] : V{};
            const V w = axpy16(wq, coef, qk);
            W[q] = w;
            acc.add(w, Qn ? qn : w);
        }
    }
    if (pa.mode == 1 && pa.k == pa.j && pa.j == pa.m) return;   // h_{m+1,m} unused
    if (pa.mode == 1) __syncwarp();    // (the sum may be formed again from what the other lanes stored)
    const double bsum = block_total(acc, red, [&](int warp) {
        const int a = pa.mode == 0 ? 0 : pa.j;
        const int b = pa.mode == 5 ? pa.k - 1 : pa.mode == 1 && pa.k < pa.j ? pa.k : a;
        return warp_dot_in_fp64(reinterpret_cast<const V*>(vptr<T>(P, a)) + q0,
                                reinterpret_cast<const V*>(vptr<T>(P, b)) + q0, (int)(q1 - q0), warp);
    });
    StageArgs a{};
    a.fin_mode = pa.mode == 0 ? (pa.notail == 2 ? FIN_NORM0_TAIL : pa.notail ? FIN_NORM0_NOTAIL : FIN_NORM0)
               : pa.mode == 7 ? FIN_STORE_NORM
               : (pa.mode == 5 ? FIN_MATVEC : FIN_MGS);
    a.fin_j = pa.j;
    a.fin_k = pa.k;
    a.m = pa.m;
    a.tol = pa.tol;
    a.partials = pa.partials;
    a.counters = pa.counters;
    partial_and_finalize_at(P, pid, a, bsum, red, &s_last, blockIdx.x, blockIdx.x - pc.y, P->pchunks);
}

// Multi-output Krylov combine (PointArgs mode 8): output q = beta sum_{k=1}^{meff} e_{q,k} s_k q_k
// for every q from one read of the basis (each output's arithmetic is that of mode 2, so an
// output equals the single combine with the same coefficients bit for bit).  A kernel of its
// own keeps the accumulators out of the flat passes' register budget.
template <typename T>
__global__ void __launch_bounds__(NTHREADS, 2)
combine_multi_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ pbase, int nprob, PointArgs pa) {
    using V = typename Vec16<T>::type;
    constexpr int NV = Vec16<T>::N;
    __shared__ T s_mc[MAX_TAU][MAX_M];
    const int2 pc = __ldg(reinterpret_cast<const int2*>(pbase + flat_block_table(nprob)) + blockIdx.x);
    const int pid = pc.x;
    const ProblemDev* P = probs + pid;
    const double* kry = P->kry;
    if (kry[KRY_NONFINITE] != 0.0 || kry[KRY_SKIP] != 0.0) return;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int meff = (int)kry[KRY_MEFF];
    const double beta = kry[KRY_BETA];
    const int nt = pa.nout + pa.final_out;
    const double* ec = pa.ecoef + (size_t)pid * nt * MAX_M;
    for (int e = tid; e < nt * meff; e += NTHREADS) {
        const int q = e / meff, k = e - q * meff;
        s_mc[q][k] = (T)(beta * ec[q * MAX_M + k] * kry[KRY_S + k + 1]);
    }
    __syncthreads();
    const long long nelem = (long long)P->nfields * P->field_stride;
    const long long e0 = (long long)pc.y * PCHUNK;
    const long long e1 = e0 + PCHUNK < nelem ? e0 + PCHUNK : nelem;
    const long long q0 = e0 / NV, q1 = e1 / NV;
    V* outs[MAX_TAU];
#pragma unroll
    for (int q = 0; q < MAX_TAU; ++q) {
        outs[q] = nullptr;
        if (q < pa.nout)
            outs[q] = pa.out ? reinterpret_cast<V*>(static_cast<T*>(pa.out) + q * pa.out_qstride +
                                                    (long long)pid * pa.out_stride)
                             : reinterpret_cast<V*>(vptr<T>(P, pa.dst + q));
        else if (q == pa.nout && pa.final_out)
            outs[q] = reinterpret_cast<V*>(vptr<T>(P, 0));
    }
    // four vectors a thread at a time (230 us one at a time, 16 shots of 401 x 201, 20 vectors)
    constexpr int G = 4;
    for (long long i = q0 + tid; i < q1; i += G * NTHREADS) {
        V acc[G][MAX_TAU];
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int q = 0; q < MAX_TAU; ++q) acc[g][q] = V{};
        for (int k = 1; k <= meff; ++k) {
            const V* B = reinterpret_cast<const V*>(vptr<T>(P, k - 1)) + i;
            V v[G];
#pragma unroll
            for (int g = 0; g < G; ++g) v[g] = i + g * NTHREADS < q1 ? B[g * NTHREADS] : V{};
#pragma unroll
            for (int q = 0; q < MAX_TAU; ++q) {
                if (q >= nt) break;
                const T c = s_mc[q][k - 1];
#pragma unroll
                for (int g = 0; g < G; ++g) fma16(acc[g][q], c, v[g]);
            }
        }
#pragma unroll
        for (int q = 0; q < MAX_TAU; ++q) {
            if (q >= nt) break;
#pragma unroll
            for (int g = 0; g < G; ++g)
                if (i + g * NTHREADS < q1) outs[q][i + g * NTHREADS] = acc[g][q];
        }
    }
}

// ---------------------------------------------------------------- Hessenberg exponential
// [13/13] Pade approximant with scaling and squaring (Higham 2005), FP64, one block per
// problem; writes exp(H_meff) e_1 to kry[KRY_E..].  Shared memory: 8 matrices of meff^2.
// One SM works alone here, at 16 cycles an FP64 warp instruction: scalar work (norm, scaling, pivot
// search, the pivot's reciprocal) is done by one warp and not by all of them, the coefficients are
// constants, products run in four interleaved sums, and Gauss-Jordan elimination takes the
// place of the serial back substitution.
struct PadeCoefs {
    double b[14];      // b_k = (26-k)! 13! / (26! k! (13-k)!)
    constexpr PadeCoefs() : b{} {
        double f[27] = {1.0};
        for (int i = 1; i <= 26; ++i) f[i] = f[i - 1] * (double)i;
        for (int k = 0; k <= 13; ++k) b[k] = f[26 - k] * f[13] / (f[26] * f[k] * f[13 - k]);
    }
};
constexpr int EXPM_THREADS = 512;

// sum_k a[k as] b[k bs], k < n
__device__ __forceinline__ double dot_strided(const double* a, int as, const double* b, int bs, int n) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    int k = 0;
    for (; k + 3 < n; k += 4)
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] = fma(a[(k + q) * as], b[(k + q) * bs], s[q]);
    for (; k < n; ++k) s[0] = fma(a[k * as], b[k * bs], s[0]);
    return (s[0] + s[1]) + (s[2] + s[3]);
}
__device__ void mat_mul(const double* A, const double* B, double* C, int n) {
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        const int r = e / n, c = e - r * n;
        C[e] = dot_strided(A + r * n, 1, B + c, n, n);
    }
    __syncthreads();
}

// Block (p, q) writes exp(tau_q H_meff) e_1 of problem p to kry[KRY_E..] (et.out null, one
// tau) or to et.out[(p ntau + q) MAX_M ..] (several taus in one launch).
__global__ void __launch_bounds__(EXPM_THREADS) expm_kernel(const ProblemDev* probs, int nprob, ExpmTaus et) {
    extern __shared__ double sm[];
    __shared__ double colsum[MAX_M];
    __shared__ int s_piv, s_scale;
    __shared__ double s_fac, s_inv;
    constexpr PadeCoefs pade;
    const ProblemDev* P = probs + blockIdx.x;
    double* kry = P->kry;
    const double hscale = et.tau[blockIdx.y];
    double* eo = et.out ? et.out + ((size_t)blockIdx.x * et.n + blockIdx.y) * MAX_M : kry + KRY_E;
    const int n = (int)kry[KRY_MEFF];
    if (n <= 0 || kry[KRY_NONFINITE] != 0.0) return;
    const int nn = n * n;
    double* A = sm;
    double* A2 = A + nn;
    double* A4 = A2 + nn;
    double* A6 = A4 + nn;
    double* Um = A6 + nn;
    double* Vm = Um + nn;
    double* Tm = Vm + nn;
    double* Wm = Tm + nn;
    const int tid = threadIdx.x;
    for (int e = tid; e < nn; e += blockDim.x) {
        const int r = e / n, c = e - r * n;
        A[e] = hscale * kry[KRY_H + r * MAX_M + c];   // exp(tau H_m): dense output at tau
    }
    __syncthreads();
    if (tid < n) {
        double s0 = 0.0, s1 = 0.0;
        int r = 0;
        for (; r + 1 < n; r += 2) {
            s0 += fabs(A[r * n + tid]);
            s1 += fabs(A[(r + 1) * n + tid]);
        }
        if (r < n) s0 += fabs(A[r * n + tid]);
        colsum[tid] = s0 + s1;
    }
    __syncthreads();
    if (tid < 32) {
        double nrm = fmax(tid < n ? colsum[tid] : 0.0, tid + 32 < n ? colsum[tid + 32] : 0.0);
        for (int o = 16; o > 0; o >>= 1) nrm = fmax(nrm, __shfl_xor_sync(0xffffffffu, nrm, o));
        // s = max(0, ceil(log2(norm / theta_13)))
        int sq = 0;
        for (double v = nrm; v > 5.371920351148152 && sq < 1000; v *= 0.5) ++sq;
        if (tid == 0) {
            s_scale = sq;
            s_fac = ldexp(1.0, -sq);
        }
    }
    __syncthreads();
    const int s = s_scale;
    for (int e = tid; e < nn; e += blockDim.x) A[e] *= s_fac;
    __syncthreads();
    mat_mul(A, A, A2, n);
    mat_mul(A2, A2, A4, n);
    mat_mul(A4, A2, A6, n);
    for (int e = tid; e < nn; e += blockDim.x) {
        Tm[e] = pade.b[13] * A6[e] + pade.b[11] * A4[e] + pade.b[9] * A2[e];
        Vm[e] = pade.b[12] * A6[e] + pade.b[10] * A4[e] + pade.b[8] * A2[e];
    }
    __syncthreads();
    // odd part U = A (A6 (b13 A6 + b11 A4 + b9 A2) + b7 A6 + b5 A4 + b3 A2 + b1 I), even part V alike
    for (int e = tid; e < 2 * nn; e += blockDim.x) {
        const bool odd = e < nn;
        const int f = odd ? e : e - nn;
        const int r = f / n, c = f - r * n;
        const double v = dot_strided(A6 + r * n, 1, (odd ? Tm : Vm) + c, n, n);
        const double a2 = A2[f], a4 = A4[f], a6 = A6[f];
        if (odd) Um[f] = v + pade.b[7] * a6 + pade.b[5] * a4 + pade.b[3] * a2 + (r == c ? pade.b[1] : 0.0);
        else Wm[f] = v + pade.b[6] * a6 + pade.b[4] * a4 + pade.b[2] * a2 + (r == c ? pade.b[0] : 0.0);
    }
    __syncthreads();
    mat_mul(A, Um, Tm, n);
    // Solve (V - U) X = (V + U): Gauss-Jordan elimination with partial pivoting; P in A2, X in A4.
    double* Pm = A2;
    double* Q = A4;
    double* mult = A6;        // multipliers of the current column
    for (int e = tid; e < nn; e += blockDim.x) {
        Pm[e] = Wm[e] - Tm[e];
        Q[e] = Wm[e] + Tm[e];
    }
    __syncthreads();
    for (int c = 0; c < n; ++c) {
        if (tid < 32) {
            double best = -1.0;
            int piv = c;
            for (int r = c + tid; r < n; r += 32) {
                const double v = fabs(Pm[r * n + c]);
                if (v > best) {
                    best = v;
                    piv = r;
                }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const double ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int op = __shfl_xor_sync(0xffffffffu, piv, o);
                if (ob > best || (ob == best && op < piv)) {
                    best = ob;
                    piv = op;
                }
            }
            if (tid == 0) {
                s_piv = piv;
                s_inv = 1.0 / Pm[piv * n + c];
            }
        }
        __syncthreads();
        const int piv = s_piv;
        const double inv = s_inv;
        // multipliers (row piv will hold what row c holds now), then the pivot row scaled into row c
        for (int r = tid; r < n; r += blockDim.x) mult[r] = r == c ? 0.0 : Pm[(r == piv ? c : r) * n + c];
        double keep_c = 0.0, keep_p = 0.0;
        const bool in_p = tid > c && tid < n, in_q = tid >= n && tid < 2 * n;
        double* M = in_p ? Pm + tid : Q + (tid - n);
        if (in_p || in_q) {
            keep_c = M[c * n];
            keep_p = M[piv * n];
        }
        __syncthreads();
        if (in_p || in_q) {
            if (piv != c) M[piv * n] = keep_c;
            M[c * n] = keep_p * inv;
        }
        __syncthreads();
        const int wp = n - c - 1, w = wp + n;      // columns c + 1 .. n - 1 of P, then all of X
        for (int e = tid; e < n * w; e += blockDim.x) {
            const int r = e / w, k = e - r * w;
            if (r == c) continue;
            double* T = k < wp ? Pm + c + 1 + k : Q + (k - wp);
            T[r * n] = fma(-mult[r], T[c * n], T[r * n]);
        }
        __syncthreads();
    }
    // X^(2^s) e_1: s - k squarings of X, then 2^k products with a vector, k by the cost of the two in
    // cycles (a squaring is bound by the FP64 pipe, 2 products a cycle; a product with a vector by
    // its latency, about 700: all 2^s of them, s = 7 for a step at 8 times the leap-frog step, were
    // half of the kernel's 200 us)
    const double cost_sq = 1500.0 + 0.6 * n * n * n, cost_mv = 700.0 + 0.6 * n * n;
    int k = 0;
    while (k < s && k < 20 && ldexp(cost_mv, k) < cost_sq) ++k;
    double* cur = Q;
    double* nxt = Um;
    for (int it = 0; it < s - k; ++it) {
        mat_mul(cur, cur, nxt, n);
        double* t = cur;
        cur = nxt;
        nxt = t;
    }
    double* x = Wm;
    double* y = Tm;
    for (int r = tid; r < n; r += blockDim.x) x[r] = (r == 0) ? 1.0 : 0.0;
    __syncthreads();
    for (int it = 0; it < 1 << k; ++it) {
        if (tid < n) y[tid] = dot_strided(cur + tid * n, 1, x, 1, n);
        __syncthreads();
        double* t = x;
        x = y;
        y = t;
    }
    if (tid < n) eo[tid] = x[tid];
}

// ---------------------------------------------------------------- Faber coefficients
// a_j = (1/N) sum_k exp(dt psi(w_k)) w_k^-j on w_k = exp(2 pi i k / N),
// psi(w) = gamma (w + c0 + c1 / w); real part:
// exp(dt gamma (c0 + (1 + c1) cos th)) cos(dt gamma (1 - c1) sin th - j th).
__global__ void faber_coeff_kernel(double dt, double gamma, double c0, double c1, int m,
                                   int N, double* out) {
    __shared__ double red[8];
    const int j = blockIdx.x;
    if (j > m) return;
    double s = 0.0;
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        const double th = 2.0 * M_PI * (double)k / (double)N;
        double sn, cs;
        sincos(th, &sn, &cs);
        const double mag = exp(dt * gamma * (c0 + (1.0 + c1) * cs));
        s += mag * cos(dt * gamma * (1.0 - c1) * sn - (double)j * th);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x / 32); ++w) t += red[w];
        out[j] = t / (double)N;
    }
}

// ---------------------------------------------------------------- launchers
void launch_set_clock(const ProblemDev* probs, int nprob, double t, double dt, cudaStream_t s) {
    set_clock_kernel<<<(nprob + 127) / 128, 128, 0, s>>>(probs, nprob, t, dt);
}
void launch_reset_cursor(const ProblemDev* probs, int nprob, cudaStream_t s) {
    reset_cursor_kernel<<<(nprob + 127) / 128, 128, 0, s>>>(probs, nprob);
}
static void launch_between(int precision, const ProblemDev* probs, int nprob, int record, int vec, int kind, int m,
                           double gamma, double c0, double c1, cudaStream_t s) {
    launch_pdl(precision == 0 ? between_kernel<float> : between_kernel<double>, nprob, PRO_THREADS, 0, s, probs, nprob,
               record, vec, kind, m, gamma, c0, c1);
}
void launch_prologue(const ProblemDev* probs, int nprob, int kind, int m, double gamma,
                     double c0, double c1, cudaStream_t s) {
    launch_between(0, probs, nprob, 0, 0, kind, m, gamma, c0, c1, s);
}
void launch_record(int precision, const ProblemDev* probs, int nprob, int vec, cudaStream_t s) {
    launch_between(precision, probs, nprob, 1, vec, -1, 0, 0.0, 0.0, 0.0, s);
}
void launch_record_next(int precision, const ProblemDev* probs, int nprob, int vec, int kind, int m, double gamma,
                        double c0, double c1, cudaStream_t s) {
    launch_between(precision, probs, nprob, 1, vec, kind, m, gamma, c0, c1, s);
}
void launch_inject(int precision, void* adj, long long vec_elems, const void* values, const int* rec, const int* nrec,
                   int nshots, int max_rec, cudaStream_t s) {
    if (precision == 0)
        inject_kernel<float><<<nshots, 256, 0, s>>>((float*)adj, vec_elems, (const float*)values, rec, nrec, max_rec);
    else
        inject_kernel<double><<<nshots, 256, 0, s>>>((double*)adj, vec_elems, (const double*)values, rec, nrec, max_rec);
}

void launch_sum_shots(int precision, const void* in, void* out, long long n, int nshots,
                      cudaStream_t s) {
    const int blocks = (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
    if (precision == 0) sum_shots_kernel<float><<<blocks, 256, 0, s>>>((const float*)in, (float*)out, n, nshots);
    else sum_shots_kernel<double><<<blocks, 256, 0, s>>>((const double*)in, (double*)out, n, nshots);
}

// Non-finite scan at the end of a step call: every block checks one PCHUNK chunk of its
// problem's state vector (the pads hold zeros) and the first block of each problem its
// Arnoldi flag; any NaN or infinity sets bit 1 (EWV error word: 1 = a pipeline wait timed
// out, 2 = a non-finite value) with one atomicOr per block that saw one.
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
nonfinite_scan_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ pbase, int nprob,
                      int* err) {
    using V = typename Vec16<T>::type;
    constexpr int NV = Vec16<T>::N;
    const int pid = flat_problem(pbase, nprob, blockIdx.x);
    const ProblemDev* P = probs + pid;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int nf = P->nfields;   // 4 (2D) or 6 (3D: w_z and psi added)
    const long long nelem = (long long)nf * P->field_stride;
    const int c = blockIdx.x - __ldg(pbase + pid);
    const long long e0 = (long long)c * PCHUNK;
    const long long e1 = e0 + PCHUNK < nelem ? e0 + PCHUNK : nelem;
    const V* S = reinterpret_cast<const V*>(vptr<T>(P, 0));
    bool bad = (c == 0 && tid == 0 && P->kry != nullptr && P->kry[KRY_NONFINITE] != 0.0);
    for (long long q = e0 / NV + tid; q < e1 / NV; q += NTHREADS) {
        const V v = S[q];
        bool b = !isfinite(v.x) || !isfinite(v.y);
        if constexpr (NV == 4) b = b || !isfinite(v.z) || !isfinite(v.w);
        bad = bad || b;
    }
    if (__syncthreads_or(bad) && tid == 0) atomicOr(err, 2);
}

void launch_nonfinite_scan(int precision, int nchunks, const ProblemDev* probs, const int* pbase,
                           int nprob, int* err, cudaStream_t s) {
    if (nchunks <= 0) return;
    const dim3 block(TPX, TPY);
    if (precision == 0) nonfinite_scan_kernel<float><<<nchunks, block, 0, s>>>(probs, pbase, nprob, err);
    else nonfinite_scan_kernel<double><<<nchunks, block, 0, s>>>(probs, pbase, nprob, err);
}

void launch_point(int precision, int nblocks, const ProblemDev* probs, const int* tile_prob,
                  const PointArgs& pa, cudaStream_t s) {
    const dim3 block(TPX, TPY);
    if (precision == 0) point_kernel<float><<<nblocks, block, 0, s>>>(probs, tile_prob, pa);
    else point_kernel<double><<<nblocks, block, 0, s>>>(probs, tile_prob, pa);
}
void launch_point_flat(int precision, int nchunks, const ProblemDev* probs, const int* pbase,
                       int nprob, const PointArgs& pa, cudaStream_t s) {
    if (nchunks <= 0) return;
    const dim3 block(TPX, TPY);
    if (pa.mode == 8) {
        if (pa.nout + pa.final_out < 1 || pa.nout + pa.final_out > MAX_TAU || !pa.ecoef) return;
        if (precision == 0) combine_multi_kernel<float><<<nchunks, block, 0, s>>>(probs, pbase, nprob, pa);
        else combine_multi_kernel<double><<<nchunks, block, 0, s>>>(probs, pbase, nprob, pa);
        return;
    }
    if (precision == 0) point_flat_kernel<float><<<nchunks, block, 0, s>>>(probs, pbase, nprob, pa);
    else point_flat_kernel<double><<<nchunks, block, 0, s>>>(probs, pbase, nprob, pa);
}
static int launch_expm_taus(const ProblemDev* probs, int nprob, int mmax, cudaStream_t s, const ExpmTaus& et) {
    const size_t smem = (size_t)8 * mmax * mmax * sizeof(double);
    if (smem > 48 * 1024) {
        if (cudaFuncSetAttribute(expm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem) != cudaSuccess)
            return -1;
    }
    expm_kernel<<<dim3(nprob, et.n), EXPM_THREADS, smem, s>>>(probs, nprob, et);
    return 0;
}
int launch_expm(const ProblemDev* probs, int nprob, int mmax, cudaStream_t s, double hscale) {
    ExpmTaus et{};
    et.n = 1;
    et.tau[0] = hscale;
    et.out = nullptr;
    return launch_expm_taus(probs, nprob, mmax, s, et);
}
int launch_expm_multi(const ProblemDev* probs, int nprob, int mmax, cudaStream_t s, const double* taus, int ntau,
                      double* out) {
    if (ntau < 1 || ntau > MAX_TAU || !out) return -1;
    ExpmTaus et{};
    et.n = ntau;
    for (int q = 0; q < ntau; ++q) et.tau[q] = taus[q];
    et.out = out;
    return launch_expm_taus(probs, nprob, mmax, s, et);
}
void launch_faber_coeffs(double dt, double gamma, double c0, double c1, int m, double* out,
                         cudaStream_t s) {
    const int N = (4 * m > 64) ? 4 * m : 64;
    faber_coeff_kernel<<<m + 1, 256, 0, s>>>(dt, gamma, c0, c1, m, N, out);
}

}  // namespace ewv
