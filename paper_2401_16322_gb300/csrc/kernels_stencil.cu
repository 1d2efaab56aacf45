// Fused stencil kernels: one HBM-streaming pass applies the operator H of Eq. (1) (or its
// transpose) to a state vector and folds in the integrator's recurrence / accumulation,
// so that every Faber degree, HORK/RK stage and Krylov matrix-vector product is one pass.
//
// Operator (Eq. 1, Sec. 2): for U = (u, v, w_x, w_y)
//   (HU)_u   = v
//   (HU)_v   = -bx by u + c^2 (u_xx + u_yy) - (bx + by) v + c^2 (d_x w_x + d_y w_y)
//   (HU)_w_x = (by - bx) d_x u - bx w_x         at (i+1/2, j)
//   (HU)_w_y = (bx - by) d_y u - by w_y         at (i, j+1/2)
// with Sec. 2.1's staggered 8th-order first derivative (Eq. spatial_8th_1) and centred
// second derivative (Eq. spatial_8th_2, "+" between the symmetric pairs), 4th-order
// textbook tables for fd_order 4, zero extension beyond the grid, and -- with a free
// surface -- Appendix A's one-sided rows for u_yy (rows 0..3) and u_y (half rows 0..2) and
// Fornberg rows (Sec. 2.2) for d_y w_y (rows 0..3).  y is the paper's upward axis, the row
// index j grows downward: d_y u at half row j+1/2 = sum_k s_k (u_{j-k} - u_{j+1+k}) / dx.
// The damping beta comes from the model's table at half-cell distances (FP32 and FP64).
//
// Layout: one thread per grid point, blocks of 32 x 4 points cut out of the BX x BY tiles of
// the work list; every operand is read straight from global memory (a warp reads 32 adjacent
// points; the taps of neighbouring points meet in L1).  These kernels serve FP64 (everything
// but 3D) and the FP32 passes that the TMA pipelines do not take (H x on a caller's vectors,
// the bfloat16 storage experiment, the allocation-free Faber step, the exact Krylov adjoint).
// In FP64 they are bound by arithmetic: GB300 issues one FP64 warp instruction per SM in
// about 16 cycles, so a pass costs its FP64 instruction count and nothing else once every SM
// has work.  Hence: small blocks (a 101 x 101 grid covers 104 SMs; 64 x 16 tiles with four
// points a thread covered 14), damping looked up instead of evaluated, terms whose
// coefficient is zero left out (the w rows of H vanish wherever no damping acts, the
// epilogue's unused operands), and no shared memory, whose bandwidth is not the limit.
// Measured on 601 x 301 in FP64: a Faber degree 35 us (102 us with four points a thread in shared
// memory), 65 FP64 instructions a point (about 150), FP64 pipe 63 % busy; HORK 12 on 101 x 101,
// FP64: 7.7 us a pass (45 us).  FP32 on 601 x 301: H x and H^T x 12.7 us for the pair (59 us).
//
// Epilogue (StageArgs), per field f at every output point:
//   K   = cx X + ch xs (H X + sigma e_src)          (xs: per-problem scale, Krylov)
//   Y   = cu U + ck K                               -> y_out
//   ACC = ca A + cau U + cak K + cay Y + cax X      -> acc_out
#include <cuda_bf16.h>

#include <type_traits>

#include "ewave_internal.cuh"
#include "grid_barrier.cuh"
#include "pdl.cuh"

namespace ewv {

// Free-surface tables: Appendix A rows (library's own copy of the printed rationals) and
// the Fornberg d_y w_y rows computed on the host at model creation.
__constant__ double g_fs_d[4 * 9 + 3 * 8 + 4 * 8];
__constant__ float g_fs_f[4 * 9 + 3 * 8 + 4 * 8];
constexpr int FS_UYY_OFF = 0, FS_UY_OFF = 36, FS_DWY_OFF = 60;

int upload_stencil_tables(int /*order*/, const double* fs_uyy, const double* fs_uy,
                          const double* fs_dwy) {
    double d[92];
    float f[92];
    for (int i = 0; i < 36; ++i) d[FS_UYY_OFF + i] = fs_uyy[i];
    for (int i = 0; i < 24; ++i) d[FS_UY_OFF + i] = fs_uy[i];
    for (int i = 0; i < 32; ++i) d[FS_DWY_OFF + i] = fs_dwy[i];
    for (int i = 0; i < 92; ++i) f[i] = (float)d[i];
    if (cudaMemcpyToSymbol(g_fs_d, d, sizeof(d)) != cudaSuccess) return -1;
    if (cudaMemcpyToSymbol(g_fs_f, f, sizeof(f)) != cudaSuccess) return -1;
    return 0;
}

template <typename T>
__device__ __forceinline__ T fs_coef(int off) {
    if constexpr (std::is_same<T, float>::value) return g_fs_f[off];
    else return g_fs_d[off];
}

// Interior tables (Eqs. spatial_8th_1/2 for R = 4; classical 4th-order tables for R = 2).
template <typename T, int R>
__device__ __forceinline__ T STAG(int k) {
    if constexpr (R == 4) {
        return k == 0 ? T(1225.0 / 1024.0) : k == 1 ? T(-245.0 / 3072.0)
             : k == 2 ? T(49.0 / 5120.0) : T(-5.0 / 7168.0);
    } else {
        return k == 0 ? T(9.0 / 8.0) : T(-1.0 / 24.0);
    }
}
template <typename T, int R>
__device__ __forceinline__ T CENT(int k) {
    if constexpr (R == 4) {
        return k == 0 ? T(-205.0 / 72.0) : k == 1 ? T(8.0 / 5.0) : k == 2 ? T(-1.0 / 5.0)
             : k == 3 ? T(8.0 / 315.0) : T(-1.0 / 560.0);
    } else {
        return k == 0 ? T(-5.0 / 2.0) : k == 1 ? T(4.0 / 3.0) : T(-1.0 / 12.0);
    }
}

// beta0 (1 - d/delta)^2 for d <= delta, d in grid units.
template <typename T>
__device__ __forceinline__ T damp(T beta0, T inv_pml, T d, int pml) {
    if (pml <= 0) return T(0);
    const T r = T(1) - d * inv_pml;
    return (d <= T(pml)) ? beta0 * r * r : T(0);
}

// Round to the nearest bfloat16 (ties to even) and widen back: the value that a bfloat16
// store followed by a load would return.
template <typename T>
__device__ __forceinline__ T bf16_round(T v) {
    return (T)__bfloat162float(__float2bfloat16_rn((float)v));
}

template <typename T>
__device__ __forceinline__ T* vec_ptr(const ProblemDev* P, int k) {
    return k == 0 ? (T*)P->state : (T*)P->work + (long long)(k - 1) * P->vec_stride;
}

// --------------------------------------------------------------------------------------
// Operands of one grid point
// --------------------------------------------------------------------------------------
constexpr int DBX = 32, DBY = 4;                              // points (threads) per block
constexpr int DSUB_X = BX / DBX, DSUB = DSUB_X * (BY / DBY);  // blocks per tile of the work list
static_assert(BX % DBX == 0 && BY % DBY == 0, "blocks must cut the tiles evenly");

// beta at k half cells from the first ghost line: the model's table, or (the allocation-free
// step has none) the profile itself.
template <typename T>
__device__ __forceinline__ T beta_at(const ProblemDev& P, int k) {
    const T* tab;
    if constexpr (std::is_same<T, float>::value) tab = P.btab;
    else tab = P.btab64;
    if (tab) return (unsigned)k < (unsigned)P.nbtab ? __ldg(tab + k) : T(0);
    if (P.pml <= 0 || k > 2 * P.pml) return T(0);
    const T r = T(1) - T(0.5) * T(k) * (T)P.inv_pml;
    return (T)P.beta0 * r * r;
}
// Distances (in half cells) of the nodes and half points; the top has no layer under a free
// surface.
__device__ __forceinline__ int dist_xn(const ProblemDev& P, int i) { return 2 * min(i + 1, P.nx - i); }
__device__ __forceinline__ int dist_xh(const ProblemDev& P, int i) { return min(2 * i + 3, 2 * (P.nx - i) - 1); }
__device__ __forceinline__ int dist_yn(const ProblemDev& P, int j) {
    return P.fs ? 2 * (P.ny - j) : 2 * min(j + 1, P.ny - j);
}
__device__ __forceinline__ int dist_yh(const ProblemDev& P, int j) {
    return P.fs ? 2 * (P.ny - j) - 1 : min(2 * j + 3, 2 * (P.ny - j) - 1);
}
template <typename T>
struct Damping {
    T xn, yn, xh, yh;     // at the node, at (i + 1/2, j) and at (i, j + 1/2)
    bool any;             // false: the w rows of H are zero and the v row has no damping term
    __device__ __forceinline__ Damping(const ProblemDev& P, int i, int j)
        : xn(beta_at<T>(P, dist_xn(P, i))), yn(beta_at<T>(P, dist_yn(P, j))),
          xh(beta_at<T>(P, dist_xh(P, i))), yh(beta_at<T>(P, dist_yh(P, j))),
          // (by distance: a comparison of FP64 values would occupy the FP64 pipe)
          any(min(min(dist_xn(P, i), dist_xh(P, i)), min(dist_yn(P, j), dist_yh(P, j))) < 2 * P.pml) {}
};

// The grid point of this thread in sub-block `sub` of tile `lt` of its problem.
struct PointAt {
    int i, j;
    __device__ __forceinline__ PointAt(const ProblemDev& P, int lt, int sub)
        : i((lt % P.tiles_x) * BX + (sub % DSUB_X) * DBX + (int)threadIdx.x),
          j((lt / P.tiles_x) * BY + (sub / DSUB_X) * DBY + (int)threadIdx.y) {}
};

// Taps at (i, j) along the row and down the column, zero off the grid: row[R + d] = x(i + d);
// col[q] = x(base + q), base = j - R, or 0 for the free-surface rows 0..3 (BAND: the rows take
// their own code, so that the others do not issue its predicated-off FP64 instructions).  N taps
// each way; nx, ny: extent of the field along its row and column.  u and w are loaded and summed one
// after the other (both at once would not fit the registers that six blocks an SM leave).
template <typename T, int R, int N, bool BAND>
struct Taps {
    T row[N], col[N];
    __device__ __forceinline__ Taps(const T* rowf, const T* colf, int i, int j, long long pitch, int nx, int ny) {
        const int base = BAND ? 0 : j - R;
        const T* r = rowf + j * pitch + i - R;
        const T* c = colf + base * pitch + i;
        if (i >= R && i - R + N <= nx && base >= 0 && base + N <= ny) {
#pragma unroll
            for (int q = 0; q < N; ++q) {
                row[q] = r[q];
                col[q] = c[q * pitch];
            }
        } else {
#pragma unroll
            for (int q = 0; q < N; ++q) {
                row[q] = (i + q >= R && i + q < nx + R) ? r[q] : T(0);
                col[q] = (base + q >= 0 && base + q < ny) ? c[q * pitch] : T(0);
            }
        }
    }
};

// a b + c rounded once.  The forward pass spells its sums out, so that every kernel that holds it
// rounds alike: a chained step gives the bits of the same step launched pass by pass.
__device__ __forceinline__ float mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return __fma_rn(a, b, c); }

// Sums of u at (i, j): the Laplacian (times dx^2) and the half-point differences d_x u at
// (i + 1/2, j), d_y u at (i, j + 1/2) (times dx).
template <typename T, int R, bool BAND>
struct USums {
    Taps<T, R, 2 * R + 1, BAND> t;
    int j;
    __device__ __forceinline__ USums(const ProblemDev& P, const T* X, int i, int jj)
        : t(X, X, i, jj, P.pitch, P.nx, P.ny), j(jj) {}
    __device__ __forceinline__ T u() const { return t.row[R]; }
    __device__ __forceinline__ T laplacian() const {
        T uxx = CENT<T, R>(0) * t.row[R], uyy;
#pragma unroll
        for (int k = 1; k <= R; ++k) uxx = mad(CENT<T, R>(k), (t.row[R + k] + t.row[R - k]), uxx);
        if constexpr (BAND) {
            uyy = T(0);
#pragma unroll
            for (int q = 0; q <= 2 * R; ++q) uyy = mad(fs_coef<T>(FS_UYY_OFF + j * 9 + q), t.col[q], uyy);
        } else {
            uyy = CENT<T, R>(0) * t.row[R];
#pragma unroll
            for (int k = 1; k <= R; ++k) uyy = mad(CENT<T, R>(k), (t.col[R + k] + t.col[R - k]), uyy);
        }
        return uxx + uyy;
    }
    __device__ __forceinline__ T du_x() const {
        T d = T(0);
#pragma unroll
        for (int k = 0; k < R; ++k) d = mad(STAG<T, R>(k), (t.row[R + 1 + k] - t.row[R - k]), d);
        return d;
    }
    __device__ __forceinline__ T du_y() const {
        T d = T(0);
        if constexpr (!BAND) {
#pragma unroll
            for (int k = 0; k < R; ++k) d = mad(STAG<T, R>(k), (t.col[R - k] - t.col[R + 1 + k]), d);
        } else if (j < 3) {
#pragma unroll
            for (int q = 0; q < 2 * R; ++q) d = mad(fs_coef<T>(FS_UY_OFF + j * 8 + q), t.col[q], d);
        } else {     // row 3: the interior stencil, counted from row 0
#pragma unroll
            for (int k = 0; k < R; ++k) d = mad(STAG<T, R>(k), (t.col[R - 1 - k] - t.col[R + k]), d);
        }
        return d;
    }
};

// (d_x w_x + d_y w_y) dx at the node: w_x[i+k] - w_x[i-1-k] and (upward y) w_y[j-1-k] - w_y[j+k];
// w_x has nx - 1 columns, w_y ny - 1 rows.
template <typename T, int R, bool BAND>
__device__ __forceinline__ T divergence(const ProblemDev& P, const T* X, int i, int j) {
    const Taps<T, R, 2 * R, BAND> t(X + 2 * P.field_stride, X + 3 * P.field_stride, i, j, P.pitch, P.nx - 1, P.ny - 1);
    T dwx = T(0), dwy = T(0);
#pragma unroll
    for (int k = 0; k < R; ++k) dwx = mad(STAG<T, R>(k), (t.row[R + k] - t.row[R - 1 - k]), dwx);
    if constexpr (BAND) {
#pragma unroll
        for (int q = 0; q < 2 * R; ++q) dwy = mad(fs_coef<T>(FS_DWY_OFF + j * 8 + q), t.col[q], dwy);
    } else {
#pragma unroll
        for (int k = 0; k < R; ++k) dwy = mad(STAG<T, R>(k), (t.col[R - 1 - k] - t.col[R + k]), dwy);
    }
    return dwx + dwy;
}

// --------------------------------------------------------------------------------------
// Epilogue of one point (StageArgs): terms whose coefficient is zero or one, or whose operand
// is absent, cost nothing.  The host sets the bits (stage_terms); the bits of the FP64 integrators
// are compile-time constants (TERMS >= 0), because a term that is skipped by predication still
// occupies the FP64 pipe.  hw: the w components of H X are not zero.
// --------------------------------------------------------------------------------------
enum { TERM_CX = 1, TERM_CK = 2, TERM_CU = 4, TERM_CA = 8, TERM_CAU = 16, TERM_CAK = 32, TERM_CAY = 64,
       TERM_CAX = 128, TERM_XS = 256, TERM_A = 512 };

static int stage_terms(const StageArgs& a) {
    int t = 0;
    if (a.cx != 0.0) t |= TERM_CX;
    if (a.ck != 1.0) t |= TERM_CK;                         // a factor other than one
    if (a.u >= 0 && a.cu != 0.0) t |= TERM_CU;
    if (a.a >= 0) t |= TERM_A;
    if (a.a >= 0 && a.ca != 1.0) t |= TERM_CA;             // ... also zero: A is read, as before
    if (a.u >= 0 && a.cau != 0.0) t |= TERM_CAU;
    if (a.cak != 0.0) t |= TERM_CAK;
    if (a.cay != 0.0) t |= TERM_CAY;
    if (a.cax != 0.0) t |= TERM_CAX;
    if (a.x_scale_slot >= 0) t |= TERM_XS;
    return t;
}

template <typename T, int TERMS>
__device__ __forceinline__ void epilogue(const ProblemDev& P, const StageArgs& a, long long o, const T (&xf)[4],
                                         const T (&hf)[4], bool hw, bool padx, bool pady) {
    const int t = TERMS >= 0 ? TERMS : a.terms;
    const T* U = (t & (TERM_CU | TERM_CAU)) ? vec_ptr<T>(&P, a.u) + o : nullptr;
    const T* A = (t & TERM_A) ? vec_ptr<T>(&P, a.a) + o : nullptr;
    T* Y = a.y_out >= 0 ? vec_ptr<T>(&P, a.y_out) + o : nullptr;
    T* ACC = a.acc_out >= 0 ? vec_ptr<T>(&P, a.acc_out) + o : nullptr;
    T uv[4], av[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        uv[f] = U ? U[f * P.field_stride] : T(0);
        av[f] = A ? A[f * P.field_stride] : T(0);
    }
    T cx = (T)a.cx, ch = (T)a.ch, cax = (T)a.cax;
    if (t & TERM_XS) {
        const T xs = (T)P.kry[a.x_scale_slot];
        cx *= xs;
        ch *= xs;
        cax *= xs;
    }
    pdl_trigger();
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        const bool pad = (f == 2 && padx) || (f == 3 && pady);
        T kf;
        if (f < 2 || hw) {
            kf = ch * hf[f];
            if (t & TERM_CX) kf = mad(cx, xf[f], kf);
        } else {
            kf = (t & TERM_CX) ? cx * xf[f] : T(0);
        }
        T yf = (t & TERM_CK) ? (T)a.ck * kf : kf;
        if (t & TERM_CU) yf = mad((T)a.cu, uv[f], yf);
        if (pad) yf = T(0);
        if (a.store_bf16) yf = bf16_round(yf);     // storage-precision experiment
        if (Y) Y[f * P.field_stride] = yf;
        if (ACC) {
            T af = (t & TERM_CA) ? (T)a.ca * av[f] : av[f];
            if (t & TERM_CAY) af = mad((T)a.cay, yf, af);
            if (t & TERM_CAU) af = mad((T)a.cau, uv[f], af);
            if (t & TERM_CAK) af = mad((T)a.cak, kf, af);
            if (t & TERM_CAX) af = mad(cax, xf[f], af);
            if (a.store_bf16) af = bf16_round(af);
            ACC[f * P.field_stride] = pad ? T(0) : af;
        }
    }
}

// --------------------------------------------------------------------------------------
// Stage kernels: one point of the forward pass, the gradient pass, the transposed pass
// --------------------------------------------------------------------------------------
enum { PASS_FORWARD = 0, PASS_GRADIENT = 1, PASS_TRANSPOSE = 2 };

template <typename T, int R, bool BAND, int TERMS>
__device__ __forceinline__ void forward_point(const ProblemDev& P, const StageArgs& a, int i, int j,
                                              const Damping<T>& b, T c2) {
    const int nx = P.nx, ny = P.ny;
    const long long o = (long long)j * P.pitch + i;
    const T* X = vec_ptr<T>(&P, a.x);
    const T idx1 = (T)P.inv_dx, idx2 = (T)P.inv_dx2;
    const bool padx = i >= nx - 1, pady = j >= ny - 1;
    const T xv = X[P.field_stride + o];
    const T xwx = padx ? T(0) : X[2 * P.field_stride + o], xwy = pady ? T(0) : X[3 * P.field_stride + o];
    T xu, lap, damping = T(0), hwx = T(0), hwy = T(0);
    {
        const USums<T, R, BAND> s(P, X, i, j);
        xu = s.u();
        lap = s.laplacian();
        if (b.any) {
            damping = -mad(b.xn * b.yn, xu, (b.xn + b.yn) * xv);
            hwx = mad((b.yn - b.xh) * idx1, s.du_x(), -(b.xh * xwx));
            hwy = mad((b.xn - b.yh) * idx1, s.du_y(), -(b.yh * xwy));
        }
    }
    if (i == P.src_i && j == P.src_j && a.src_slot >= 0 && P.has_src) damping += (T)P.sigma[a.src_slot];
    const T hv = mad(c2, mad(lap, idx2, divergence<T, R, BAND>(P, X, i, j) * idx1), damping);
    const T xf[4] = {xu, xv, xwx, xwy}, hf[4] = {xv, hv, hwx, hwy};
    epilogue<T, TERMS>(P, a, o, xf, hf, b.any, padx, pady);
}

// FWI gradient with respect to m = c^2: grad += gscale q_v xs (L X_u + D X_w) = gscale q_v d(H X)_v/dm
template <typename T, int R, bool BAND>
__device__ __forceinline__ void gradient_point(const ProblemDev& P, const StageArgs& a, int i, int j) {
    const long long o = (long long)j * P.pitch + i;
    const T* X = vec_ptr<T>(&P, a.x);
    T* G = static_cast<T*>(a.grad) + (long long)P.shot * P.field_stride;
    const T xs = a.x_scale_slot >= 0 ? (T)P.kry[a.x_scale_slot] : T(1);
    const T g = USums<T, R, BAND>(P, X, i, j).laplacian() * (T)P.inv_dx2 + divergence<T, R, BAND>(P, X, i, j) * (T)P.inv_dx;
    G[o] += (T)a.gscale * xs * vec_ptr<T>(&P, a.gq)[P.field_stride + o] * g;
}

// H^T y from y (unscaled): z_v = c^2 y_v, z_x = (by - bx^h) y_wx, z_y = (bx - by^h) y_wy.
template <typename T, int R, int TERMS>
__device__ __forceinline__ void transpose_point(const ProblemDev& P, const StageArgs& a, int i, int j) {
    const int nx = P.nx, ny = P.ny;
    const bool fs = P.fs != 0;
    const long long pitch = P.pitch, o = j * pitch + i;
    const T* X = vec_ptr<T>(&P, a.x);
    const T* Xv = X + P.field_stride;
    const T* Xwx = X + 2 * P.field_stride;
    const T* Xwy = X + 3 * P.field_stride;
    const T* C2 = static_cast<const T*>(P.c2);
    const T idx1 = (T)P.inv_dx, idx2 = (T)P.inv_dx2;
    const bool padx = i >= nx - 1, pady = j >= ny - 1;
    const T xu = X[o], xv = Xv[o], xwx = padx ? T(0) : Xwx[o], xwy = pady ? T(0) : Xwy[o];
    const Damping<T> b(P, i, j);
    T zx[2 * R + 1], zy[2 * R + 1];           // z_v along the row and down the column
#pragma unroll
    for (int q = 0; q <= 2 * R; ++q) {
        const int c = i + q - R, r = j + q - R;
        zx[q] = (c >= 0 && c < nx) ? C2[o + q - R] * Xv[o + q - R] : T(0);
        const long long p = o + (q - R) * pitch;
        zy[q] = (r >= 0 && r < ny) ? C2[p] * Xv[p] : T(0);
    }
    // (Lxx^T z_v)(i) = Lxx z_v; (Lyy^T z_v)(j): rows r >= rfs contribute CENT(|r - j|), the
    // free-surface rows r < 4 FS_UYY[r][j] for j <= 8
    T lxx = CENT<T, R>(0) * zx[R], lyy = T(0);
#pragma unroll
    for (int k = 1; k <= R; ++k) lxx += CENT<T, R>(k) * (zx[R + k] + zx[R - k]);
    const int rfs = fs ? 4 : 0;
#pragma unroll
    for (int k = -R; k <= R; ++k)
        if (j + k >= rfs) lyy += CENT<T, R>(k < 0 ? -k : k) * zy[R + k];
    // (Dxn^T z_v)(i+1/2) = sum_k s_k (z_v[i-k] - z_v[i+1+k]); (Dyn^T z_v)(j+1/2) with the rows'
    // s_k (w[r-1-k] - w[r+k]), the free-surface rows r < 4 FS_DWY[r][j] for j <= 7
    T dxt = T(0), dyt = T(0);
#pragma unroll
    for (int k = 0; k < R; ++k) dxt += STAG<T, R>(k) * (zx[R - k] - zx[R + 1 + k]);
#pragma unroll
    for (int k = 0; k < R; ++k) {
        if (j + 1 + k >= rfs) dyt += STAG<T, R>(k) * zy[R + 1 + k];
        if (j - k >= rfs) dyt -= STAG<T, R>(k) * zy[R - k];
    }
    if (fs && j <= 8) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (r >= ny) break;
            const T z = C2[r * pitch + i] * Xv[r * pitch + i];
            lyy += fs_coef<T>(FS_UYY_OFF + r * 9 + j) * z;
            if (j <= 7) dyt += fs_coef<T>(FS_DWY_OFF + r * 8 + j) * z;
        }
    }
    // (Dxh^T z_x)(i) = sum_k s_k (z_x[i-1-k] - z_x[i+k]), the half columns i-R .. i+R-1 (beta
    // falls towards the middle: none damps unless one of the two ends does)
    T gxt = T(0), gyt = T(0);
    if (min(dist_yn(P, j), min(dist_xh(P, max(i - R, 0)), dist_xh(P, min(i + R - 1, nx - 2)))) < 2 * P.pml) {
#pragma unroll
        for (int q = 0; q < 2 * R; ++q) {
            const int p = i - R + q;
            if (p < 0 || p >= nx - 1) continue;
            const T z = (b.yn - beta_at<T>(P, dist_xh(P, p))) * Xwx[o + q - R];
            gxt += (q < R ? STAG<T, R>(R - 1 - q) : -STAG<T, R>(q - R)) * z;
        }
    }
    // (Dyh^T z_y)(j): half rows h >= hfs of d_y u use s_k (u[h-k] - u[h+1+k]), the
    // free-surface half rows h < 3 FS_UY[h][j] for j <= 7
    if ((fs && j <= 7) ||
        min(dist_xn(P, i), min(dist_yh(P, max(j - R, 0)), dist_yh(P, min(j + R - 1, ny - 2)))) < 2 * P.pml) {
        const int hfs = fs ? 3 : 0;
#pragma unroll
        for (int q = 0; q < 2 * R; ++q) {
            const int h = j - R + q;
            if (h < hfs || h >= ny - 1) continue;
            const T z = (b.xn - beta_at<T>(P, dist_yh(P, h))) * Xwy[o + (q - R) * pitch];
            gyt += (q < R ? -STAG<T, R>(R - 1 - q) : STAG<T, R>(q - R)) * z;
        }
        if (fs && j <= 7) {
#pragma unroll
            for (int h = 0; h < 3; ++h)
                if (h < ny - 1)
                    gyt += fs_coef<T>(FS_UY_OFF + h * 8 + j) *
                           ((b.xn - beta_at<T>(P, dist_yh(P, h))) * Xwy[h * pitch + i]);
        }
    }
    const T xf[4] = {xu, xv, xwx, xwy};
    const T hf[4] = {-b.xn * b.yn * xv + (lxx + lyy) * idx2 + (gxt + gyt) * idx1, xu - (b.xn + b.yn) * xv,
                     padx ? T(0) : dxt * idx1 - b.xh * xwx, pady ? T(0) : dyt * idx1 - b.yh * xwy};
    epilogue<T, TERMS>(P, a, o, xf, hf, true, padx, pady);
}

template <typename T, int R, int PASS, int TERMS>
__device__ __forceinline__ void stage_point(const ProblemDev& P, const StageArgs& a, int lt, int sub) {
    const PointAt q(P, lt, sub);
    pdl_wait();
    if (q.i >= P.nx || q.j >= P.ny) return;
    const bool band = R == 4 && P.fs != 0 && q.j < 4;       // (a warp is one row)
    if constexpr (PASS == PASS_FORWARD) {
        const Damping<T> b(P, q.i, q.j);
        const T c2 = static_cast<const T*>(P.c2)[(long long)q.j * P.pitch + q.i];
        if (band) forward_point<T, R, R == 4, TERMS>(P, a, q.i, q.j, b, c2);
        else forward_point<T, R, false, TERMS>(P, a, q.i, q.j, b, c2);
    } else if constexpr (PASS == PASS_GRADIENT) {
        if (band) gradient_point<T, R, R == 4>(P, a, q.i, q.j);
        else gradient_point<T, R, false>(P, a, q.i, q.j);
    } else {
        transpose_point<T, R, TERMS>(P, a, q.i, q.j);
    }
}

// Every problem of an engine through its tile work list.
template <typename T, int R, int PASS, int TERMS>
__global__ void __launch_bounds__(DBX * DBY, 6)
stage_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ tile_prob, StageArgs a) {
    const int tile = blockIdx.x / DSUB;
    const ProblemDev& P = probs[tile_prob[tile]];
    stage_point<T, R, PASS, TERMS>(P, a, tile - P.tile_base, blockIdx.x % DSUB);
}

// One problem whose descriptor travels with the launch (H x on a caller's vectors: no device
// copy of the descriptor to allocate, fill and wait for).
template <typename T, int R, int PASS, int TERMS>
__global__ void __launch_bounds__(DBX * DBY, 6)
stage_one_kernel(const __grid_constant__ ProblemDev P, StageArgs a) {
    stage_point<T, R, PASS, TERMS>(P, a, blockIdx.x / DSUB, blockIdx.x % DSUB);
}

// --------------------------------------------------------------------------------------
// The passes of one step in one cooperative launch (FP64, small grids).  A thread keeps its point
// through all of them (damping, c^2 and descriptor stay in registers) and a bounded grid barrier
// takes the place of the launch between two passes: at a few blocks per SM a pass computes for 2 to
// 8 us, and setting a kernel up and draining it costs more than the barrier.  us a pass, launched
// one by one and chained: HORK 8.5 -> 6.8 on 101 x 101, 11.5 -> 9.2 on 150 x 150, 13.8 -> 11.1 on
// 250 x 200, 17.3 -> 13.1 on 251 x 251 (Faber and the Horner form likewise); HORK 12, 4th order,
// 101 x 101, 4 steps: 367 -> 297 us.
// bar: [0] arrivals, [1] blocks that have left; the last one clears both for the next launch.
// --------------------------------------------------------------------------------------
__device__ unsigned long long g_chain_wait_limit_ns = 1000000000ull;

int set_chain_wait_limit_ns(unsigned long long ns) {
    return cudaMemcpyToSymbol(g_chain_wait_limit_ns, &ns, sizeof(ns)) == cudaSuccess ? 0 : -1;
}

template <typename T, int R, int TERMS>
__global__ void __launch_bounds__(DBX * DBY, 4)
chain_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ tile_prob,
             const __grid_constant__ PassChain chain, unsigned int* bar, int* err) {
    __shared__ int s_ok;
    const unsigned long long lim = g_chain_wait_limit_ns;
    const int tile = blockIdx.x / DSUB;
    const ProblemDev P = probs[tile_prob[tile]];
    const PointAt q(P, tile - P.tile_base, blockIdx.x % DSUB);
    const bool in = q.i < P.nx && q.j < P.ny, band = R == 4 && P.fs != 0 && q.j < 4;
    const Damping<T> b(P, q.i, q.j);
    const T c2 = in ? static_cast<const T*>(P.c2)[(long long)q.j * P.pitch + q.i] : T(0);
    for (int n = 0; n < chain.n; ++n) {
        const StageArgs a = chain_stage(chain.pass[n]);
        if (in) {
            if (a.terms == TERMS) {
                if (band) forward_point<T, R, R == 4, TERMS>(P, a, q.i, q.j, b, c2);
                else forward_point<T, R, false, TERMS>(P, a, q.i, q.j, b, c2);
            } else {
                if (band) forward_point<T, R, R == 4, -1>(P, a, q.i, q.j, b, c2);
                else forward_point<T, R, false, -1>(P, a, q.i, q.j, b, c2);
            }
        }
        if (n + 1 < chain.n && !grid_phase_barrier(bar, (unsigned)(n + 1), lim, &s_ok)) {
            if (threadIdx.x == 0 && threadIdx.y == 0) atomicOr(err, 1);
            break;
        }
    }
    chain_leave(bar);
}

// --------------------------------------------------------------------------------------
// Leap-frog step in FP64 (Sec. 3.1).  Vectors `cur` (u^n, w^n) and `prev` (u^{n-1}, w^{n-1}) use
// fields 0 (u), 2 (w_x), 3 (w_y); level n+1 overwrites `prev`.  Variant 2 (difference form)
// reads d^n = u^n - u^{n-1} from field 1 of `prev` instead of u^{n-1} and writes d^{n+1} to
// field 1 of `cur` (read by no other thread of the step), u^{n+1} = u^n + d^{n+1}.
// Where nothing damps, the w fields keep their level n-1 values and u^{n+1} needs no division
// (an FP64 division costs as much as half the stencil).
// --------------------------------------------------------------------------------------
template <typename T, int R, bool BAND>
__device__ __forceinline__ void leapfrog_point(const ProblemDev& P, int i, int j, int cur, int prev, int variant,
                                               double dt_d) {
    const int nx = P.nx, ny = P.ny;
    const long long fstr = P.field_stride, o = (long long)j * P.pitch + i;
    T* Cn = vec_ptr<T>(&P, cur);
    T* Pn = vec_ptr<T>(&P, prev);
    const T dt = (T)dt_d, idx1 = (T)P.inv_dx, idx2 = (T)P.inv_dx2;
    const bool inx = i < nx - 1, iny = j < ny - 1;
    const T um = Pn[(variant == 2 ? fstr : 0) + o];
    const T wxm = inx ? Pn[2 * fstr + o] : T(0), wym = iny ? Pn[3 * fstr + o] : T(0);
    const T c2 = static_cast<const T*>(P.c2)[o];
    const Damping<T> b(P, i, j);
    const T wx = inx ? Cn[2 * fstr + o] : T(0), wy = iny ? Cn[3 * fstr + o] : T(0);
    T u, lap, gx = T(0), gy = T(0);
    {
        const USums<T, R, BAND> s(P, Cn, i, j);
        u = s.u();
        lap = s.laplacian();
        if (b.any) {
            gx = (b.yn - b.xh) * s.du_x() * idx1;
            gy = (b.xn - b.yh) * s.du_y() * idx1;
        }
    }
    T rhs = c2 * (lap * idx2 + divergence<T, R, BAND>(P, Cn, i, j) * idx1);
    if (i == P.src_i && j == P.src_j && P.has_src) rhs += (T)P.sigma[0];
    T up, wxp = wxm, wyp = wym;
    if (!b.any) {
        if (variant == 2) {
            const T dn = um + dt * dt * rhs;
            Cn[fstr + o] = dn;
            up = u + dn;
        } else {
            up = (T(2) * u - um) + dt * dt * rhs;
        }
    } else {
        const T bsum = b.xn + b.yn;
        rhs -= b.xn * b.yn * u;
        if (variant == 2) {
            // (u^{n+1} - u^n)(1 + b dt/2) = d^n (1 - b dt/2) + dt^2 rhs, with d^n = um
            const T hb = T(0.5) * bsum * dt;
            const T dn = (um * (T(1) - hb) + dt * dt * rhs) / (T(1) + hb);
            Cn[fstr + o] = dn;
            up = u + dn;
        } else {
            const T inv_dt2 = T(1) / (dt * dt), inv_2dt = T(1) / (T(2) * dt);
            up = ((T(2) * u - um) * inv_dt2 + bsum * um * inv_2dt + rhs) / (inv_dt2 + bsum * inv_2dt);
        }
        if (inx)
            wxp = variant != 1 ? ((T(1) - b.xh * dt) * wxm + T(2) * dt * gx) / (T(1) + b.xh * dt)
                               : wxm + T(2) * dt * (-b.xh * wx + gx);
        if (iny)
            wyp = variant != 1 ? ((T(1) - b.yh * dt) * wym + T(2) * dt * gy) / (T(1) + b.yh * dt)
                               : wym + T(2) * dt * (-b.yh * wy + gy);
    }
    pdl_trigger();
    Pn[o] = up;
    Pn[2 * fstr + o] = wxp;
    Pn[3 * fstr + o] = wyp;
}

template <typename T, int R>
__global__ void __launch_bounds__(DBX * DBY, 6)
leapfrog_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ tile_prob,
                int cur, int prev, int variant, double dt) {
    const int tile = blockIdx.x / DSUB;
    const ProblemDev& P = probs[tile_prob[tile]];
    const PointAt q(P, tile - P.tile_base, blockIdx.x % DSUB);
    pdl_wait();
    if (q.i >= P.nx || q.j >= P.ny) return;
    if (R == 4 && P.fs != 0 && q.j < 4) leapfrog_point<T, R, R == 4>(P, q.i, q.j, cur, prev, variant, dt);
    else leapfrog_point<T, R, false>(P, q.i, q.j, cur, prev, variant, dt);
}

// --------------------------------------------------------------------------------------
template <int V>
using Int = std::integral_constant<int, V>;

// Calls launch(T(), Int<R>, Int<PASS>) for the pass that `a` asks for.
template <int PASS, class F>
static void with_type(int precision, int R, F&& launch) {
    if (precision == 0 && R == 4) launch(float(), Int<4>(), Int<PASS>());
    else if (precision == 0) launch(float(), Int<2>(), Int<PASS>());
    else if (R == 4) launch(double(), Int<4>(), Int<PASS>());
    else launch(double(), Int<2>(), Int<PASS>());
}
template <class F>
static void with_pass(int precision, int R, const StageArgs& a, F&& launch) {
    if (a.transpose) with_type<PASS_TRANSPOSE>(precision, R, launch);
    else if (a.grad) with_type<PASS_GRADIENT>(precision, R, launch);
    else with_type<PASS_FORWARD>(precision, R, launch);
}

// Programmatic dependent launch from about four blocks per SM on, which is where chained steps end
// too.  us a pass in FP64, dependent and plain: Faber 19.5 and 19.9 at 640 blocks (300 x 250), 22.7 and
// 22.7 at 912, 27.7 and 28.2 at 1120, 33.4 and 33.9 at 1520 (601 x 301), 54.4 and 54.9 at 2704; Horner
// HORK 17.1 and 17.6, 19.4 and 19.8, 23.6 and 24.1, 27.9 and 28.6, 44.5 and 45.0; H x 14.9 and 16.7,
// 16.9 and 18.8, 21.1 and 23.2, 25.0 and 27.1, 40.6 and 43.2.  It loses at single sizes only (Faber and
// low-storage HORK at 680 blocks, by 2 and 4 %; the leap-frog step at 912, by 6 %).  A grid of a block
// per SM or less ran slower that way (112 blocks of 101 x 101: 7.7 -> 8.2 us a pass), its blocks set
// up early end up sharing SMs.
template <class... P, class... A>
static void launch_plain(void (*kernel)(P...), int blocks, cudaStream_t s, A... args) {
    const dim3 block(DBX, DBY);
    if (blocks >= 600) launch_pdl(kernel, blocks, block, 0, s, args...);
    else kernel<<<blocks, block, 0, s>>>(static_cast<P>(args)...);
}

void launch_stage(int precision, int R, int ntiles, const ProblemDev* probs, const int* tile_prob,
                  const StageArgs& a_in, cudaStream_t s) {
    if (ntiles <= 0) return;
    StageArgs a = a_in;
    a.terms = stage_terms(a);
    with_pass(precision, R, a, [&](auto zero, auto r, auto pass) {
        using T = decltype(zero);
        constexpr int RR = decltype(r)::value, PASS = decltype(pass)::value;
        const int blocks = ntiles * DSUB;
        if constexpr (sizeof(T) == 8 && PASS == PASS_FORWARD) {
            constexpr int FABER = TERM_CX | TERM_CU | TERM_A | TERM_CAY, HORK = TERM_CX | TERM_A | TERM_CAY;
            switch (a.terms) {
                case FABER: launch_plain(stage_kernel<T, RR, PASS, FABER>, blocks, s, probs, tile_prob, a); return;
                case HORK: launch_plain(stage_kernel<T, RR, PASS, HORK>, blocks, s, probs, tile_prob, a); return;
                case TERM_CU: launch_plain(stage_kernel<T, RR, PASS, TERM_CU>, blocks, s, probs, tile_prob, a); return;
                case TERM_XS: launch_plain(stage_kernel<T, RR, PASS, TERM_XS>, blocks, s, probs, tile_prob, a); return;
                default: break;
            }
        }
        launch_plain(stage_kernel<T, RR, PASS, -1>, blocks, s, probs, tile_prob, a);
    });
}

// (only y = H x and y = H^T x come here: no term but the product)
int launch_stage_one(int precision, int R, const ProblemDev& P, const StageArgs& a, cudaStream_t s) {
    if (stage_terms(a) != 0 || a.grad || a.store_bf16) return -1;
    with_pass(precision, R, a, [&](auto zero, auto r, auto pass) {
        constexpr int PASS = decltype(pass)::value;
        if constexpr (PASS != PASS_GRADIENT)
            launch_plain(stage_one_kernel<decltype(zero), decltype(r)::value, PASS, 0>, P.ntiles * DSUB, s, P, a);
    });
    return 0;
}

template <typename T, int R, int TERMS>
static int launch_chain_of(int blocks, const ProblemDev* probs, const int* tile_prob, const PassChain& chain,
                           unsigned int* bar, int* err, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(DBX, DBY);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, chain_kernel<T, R, TERMS>, probs, tile_prob, chain, bar, err) == cudaSuccess ? 0 : -1;
}

// Grids whose passes are chained: up to four blocks per SM, which are co-resident for every
// instantiation (128 threads, at most 128 registers).  Chaining still gains a quarter at that size;
// larger grids (300 x 250: 20 us a pass) have no choice.
bool chain_fits(int ntiles) {
    int dev = 0, nsm = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess)
        return false;
    return coop && ntiles > 0 && ntiles * DSUB <= 4 * nsm;
}

int launch_chain(int R, int ntiles, const ProblemDev* probs, const int* tile_prob, const PassChain& chain_in,
                 unsigned int* bar, int* err, cudaStream_t s) {
    constexpr int FABER = TERM_CX | TERM_CU | TERM_A | TERM_CAY, HORK = TERM_CX | TERM_A | TERM_CAY;
    static thread_local PassChain chain;        // (13 KB: not on the caller's stack)
    chain = chain_in;
    int count[3] = {0, 0, 0};
    for (int n = 0; n < chain.n; ++n) {
        const int t = chain.pass[n].terms = stage_terms(chain_stage(chain.pass[n]));
        ++count[t == FABER ? 0 : t == HORK ? 1 : 2];
    }
    const int blocks = ntiles * DSUB;
    auto go = [&](auto r) {
        constexpr int RR = decltype(r)::value;
        if (count[0] >= count[1] && count[0] >= count[2])
            return launch_chain_of<double, RR, FABER>(blocks, probs, tile_prob, chain, bar, err, s);
        if (count[1] >= count[2])
            return launch_chain_of<double, RR, HORK>(blocks, probs, tile_prob, chain, bar, err, s);
        return launch_chain_of<double, RR, TERM_CU>(blocks, probs, tile_prob, chain, bar, err, s);
    };
    return R == 4 ? go(Int<4>()) : go(Int<2>());
}

void launch_leapfrog(int R, int ntiles, const ProblemDev* probs, const int* tile_prob, int cur, int prev,
                     int variant, double dt, cudaStream_t s) {
    if (ntiles <= 0) return;
    if (R == 4) launch_plain(leapfrog_kernel<double, 4>, ntiles * DSUB, s, probs, tile_prob, cur, prev, variant, dt);
    else launch_plain(leapfrog_kernel<double, 2>, ntiles * DSUB, s, probs, tile_prob, cur, prev, variant, dt);
}

// --------------------------------------------------------------------------------------
// Pointwise parts of the discrete adjoint of the leap-frog step (averaged damping of w).
// One step maps z^n = (u^n, u^{n-1}, w^n, w^{n-1}) to z^{n+1} with
//   u^{n+1} = s (2u^n/dt^2 + (b/(2dt) - 1/dt^2) u^{n-1} + H_vu u^n + H_vw w^n + f),
//   w^{n+1} = ((1 - beta dt) w^{n-1} + 2 dt H_wu u^n) / (1 + beta dt),
// s = 1 / (1/dt^2 + b/(2dt)), b = b_x + b_y at the node, beta the w row's own damping, and
// H_vu, H_vw, H_wu blocks of H (Eq. 1).  Its transpose needs one H^T pass on
// q = (0, s lam_u, 2 dt lam_w / (1 + beta dt)):
//   lam_u'   = (H^T q)_u + (2/dt^2) s lam_u + lam_um,
//   lam_um'  = s (b/(2dt) - 1/dt^2) lam_u,
//   lam_w'   = (H^T q)_w + beta q_w + lam_wm        ((H^T q)_w holds -beta q_w),
//   lam_wm'  = (1 - beta dt) / (1 + beta dt) lam_w.
// Layout: vector 0 of a problem holds (lam_u, lam_um, lam_wx, lam_wy) (lam_um in the v field),
// a1 + shot * vec_stride holds lam_wm in its w fields.  mode 0 writes q into vector `qv`;
// mode 1 applies the update above with (H^T q) in vector `yv`.
// --------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
leapfrog_adjoint_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ tile_prob,
                        int mode, int qv, int yv, void* a1_base, double dt_d) {
    const int pid = tile_prob[blockIdx.x];
    const ProblemDev* P = probs + pid;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int nx = P->nx, ny = P->ny, pitch = P->pitch, pml = P->pml;
    const bool fs = P->fs != 0;
    const int lt = blockIdx.x - P->tile_base;
    const int x0 = (lt % P->tiles_x) * BX, y0 = (lt / P->tiles_x) * BY;
    const long long fstr = P->field_stride;
    const T beta0 = (T)P->beta0, inv_pml = (T)P->inv_pml;
    const T dt = (T)dt_d;
    T* L0 = vec_ptr<T>(P, 0);
    T* L1 = (T*)a1_base + (long long)P->shot * P->vec_stride;
#pragma unroll
    for (int b = 0; b < VY; ++b)
#pragma unroll
        for (int c = 0; c < VX; ++c) {
            const int i = x0 + tx + c * TPX, j = y0 + ty + b * TPY;
            if (i >= nx || j >= ny) continue;
            const long long o = (long long)j * pitch + i;
            const T bxn = damp<T>(beta0, inv_pml, T(min(i + 1, nx - i)), pml);
            const T byn = damp<T>(beta0, inv_pml, fs ? T(ny - j) : T(min(j + 1, ny - j)), pml);
            const T bxh = damp<T>(beta0, inv_pml, min(T(i) + T(1.5), T(nx - i) - T(0.5)), pml);
            const T byh = damp<T>(beta0, inv_pml,
                                  fs ? (T(ny - j) - T(0.5)) : min(T(j) + T(1.5), T(ny - j) - T(0.5)),
                                  pml);
            const T bsum = bxn + byn;
            const T inv_dt2 = T(1) / (dt * dt), inv_2dt = T(1) / (T(2) * dt);
            const T sn = T(1) / (inv_dt2 + bsum * inv_2dt);
            const bool hx = i < nx - 1, hy = j < ny - 1;
            const T lu = L0[o], lwx = hx ? L0[2 * fstr + o] : T(0), lwy = hy ? L0[3 * fstr + o] : T(0);
            if (mode == 0) {
                T* Q = vec_ptr<T>(P, qv);
                Q[o] = T(0);
                Q[fstr + o] = sn * lu;
                Q[2 * fstr + o] = hx ? T(2) * dt * lwx / (T(1) + bxh * dt) : T(0);
                Q[3 * fstr + o] = hy ? T(2) * dt * lwy / (T(1) + byh * dt) : T(0);
            } else {
                const T* Y = vec_ptr<T>(P, yv);
                // every operand is loaded before the first store (one memory round trip)
                const T lum = L0[fstr + o], yu = Y[o];
                const T ywx = hx ? Y[2 * fstr + o] : T(0), l1x = hx ? L1[2 * fstr + o] : T(0);
                const T ywy = hy ? Y[3 * fstr + o] : T(0), l1y = hy ? L1[3 * fstr + o] : T(0);
                L0[o] = yu + T(2) * inv_dt2 * sn * lu + lum;
                L0[fstr + o] = sn * (bsum * inv_2dt - inv_dt2) * lu;
                if (hx) {
                    const T qx = T(2) * dt * lwx / (T(1) + bxh * dt);
                    L0[2 * fstr + o] = ywx + bxh * qx + l1x;
                    L1[2 * fstr + o] = (T(1) - bxh * dt) / (T(1) + bxh * dt) * lwx;
                }
                if (hy) {
                    const T qy = T(2) * dt * lwy / (T(1) + byh * dt);
                    L0[3 * fstr + o] = ywy + byh * qy + l1y;
                    L1[3 * fstr + o] = (T(1) - byh * dt) / (T(1) + byh * dt) * lwy;
                }
            }
        }
}

void launch_leapfrog_adjoint(int precision, int nblocks, const ProblemDev* probs, const int* tile_prob,
                             int mode, int qv, int yv, void* a1_base, double dt, cudaStream_t s) {
    const dim3 block(TPX, TPY);
    if (nblocks <= 0) return;
    if (precision == 0)
        leapfrog_adjoint_kernel<float><<<nblocks, block, 0, s>>>(probs, tile_prob, mode, qv, yv, a1_base, dt);
    else
        leapfrog_adjoint_kernel<double><<<nblocks, block, 0, s>>>(probs, tile_prob, mode, qv, yv, a1_base, dt);
}

}  // namespace ewv
