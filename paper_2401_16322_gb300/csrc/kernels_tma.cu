// Persistent, TMA-fed fused stencil pass (FP32, forward operator) for sm_103a.
//
// Same arithmetic as stage_kernel (kernels_stencil.cu: Eq. 1's operator, Sec. 2.1 stencils,
// Appendix A / Sec. 2.2 free-surface rows, in-register damping, and the
// K / Y / ACC epilogue of every integrator), organised for HBM bandwidth:
//   - one CTA per SM walks the tile work list (tiles b, b + gridDim.x, ...);
//   - the last warp (one elected lane) is the producer: for each tile it issues TMA tensor loads
//     (cp.async.bulk.tensor) of every operand into one of NST shared-memory stages and
//     arms the stage's "full" mbarrier with the transaction byte count;
//   - the other warps are consumers: they wait on "full", compute the tile from shared memory
//     (two adjacent columns and one to four rows per thread), store Y / ACC with coalesced
//     st.global, and arrive on the stage's "empty" mbarrier.
// The TMA boxes (4D tensor maps over x, y, field, vector) start R rows above and 4 columns
// left of the tile (16-byte aligned x); out-of-range elements are filled with zeros by
// the TMA unit, which is exactly the zero extension of Sec. 2.1.
// Every mbarrier wait is bounded (1 s of %globaltimer): on expiry the kernel records an
// error word, drains its own outstanding copies (bounded) and returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <vector>

#include "ewave_internal.cuh"
#include "pdl.cuh"

namespace ewv {

constexpr int TX = 4;                 // staged x halo (>= R, keeps the box start 16-B aligned)
constexpr int NMAP = 12;              // tensor maps per problem and tile height

// Shared-memory layout of one stage (floats) for tile height BYv; every buffer starts on a
// 128-byte boundary.  HASU = false drops the U buffer (passes without a U operand, e.g. the
// HORK stages) and HASA = false the A buffer (passes without an A operand: the Horner HORK
// passes, the Krylov products), so that more stages or taller tiles fit in shared memory.
template <int R, int BYv, bool HASU = true, bool HASA = true>
struct StageLayout {
    static constexpr int up32(int v) { return (v + 31) / 32 * 32; }   // 128-byte boundary
    static constexpr int SH = BYv + 2 * R;
    static constexpr int SW = BX + 2 * TX;
    static constexpr int U_OFF = 0;                                // u      SH x SW
    static constexpr int WX_OFF = up32(U_OFF + SH * SW);           // w_x    BYv x SW
    static constexpr int WY_OFF = up32(WX_OFF + BYv * SW);         // w_y    SH x BX
    static constexpr int V_OFF = WY_OFF + SH * BX;                 // v      BYv x BX
    static constexpr int C2_OFF = V_OFF + BYv * BX;                // c^2    BYv x BX
    static constexpr int PU_OFF = C2_OFF + BYv * BX;               // U      4 x BYv x BX
    static constexpr int PA_OFF = PU_OFF + (HASU ? 4 * BYv * BX : 0);   // A  4 x BYv x BX
    static constexpr int FLOATS = PA_OFF + (HASA ? 4 * BYv * BX : 0);
    // floats the five field boxes deliver (the padding between buffers is not written)
    static constexpr int BOX_FLOATS = SH * SW + BYv * SW + SH * BX + 2 * BYv * BX;
    static constexpr int BYTES = FLOATS * 4;
    static_assert((U_OFF * 4) % 128 == 0 && (WX_OFF * 4) % 128 == 0 && (WY_OFF * 4) % 128 == 0 &&
                      (V_OFF * 4) % 128 == 0 && (C2_OFF * 4) % 128 == 0 &&
                      (PU_OFF * 4) % 128 == 0 && (PA_OFF * 4) % 128 == 0 && BYTES % 128 == 0,
                  "TMA destinations must be 128-byte aligned");
};

// What the producer resolves once per tile and hands to the consumers with the stage.
struct __align__(16) TileInfo {
    float* Y;
    float* A;
    float* T;                // field of the gradient tape (adjoint steps), or null
    float* G;                // this shot's gradient field, or null
    long long fstr;
    int x0, y0, nx, ny, pitch, pml, fs, src_i, src_j, shot;
    float beta0, inv_pml, idx1, idx2, sig, xs;   // xs: per-problem scale of H X (Krylov)
    const float* btab;       // damping at half-cell distances (ProblemDev::btab)
    int nbtab;
    int xdamp;               // the tile's columns, and 8 more on each side, touch the damping layer
};

// The consumers read a stage's TileInfo with 16-byte shared loads into registers.
__device__ __forceinline__ TileInfo load_info(const TileInfo* p) {
    static_assert(sizeof(TileInfo) % 16 == 0, "TileInfo must be a whole number of 16-byte words");
    union {
        TileInfo t;
        int4 v[sizeof(TileInfo) / 16];
    } u;
#pragma unroll
    for (int q = 0; q < (int)(sizeof(TileInfo) / 16); ++q) u.v[q] = reinterpret_cast<const int4*>(p)[q];
    return u.t;
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Limit of the pipeline waits (ns).  1 s by default; ewv_debug_set_wait_limit lowers it so
// that a test can make a wait give up on a healthy GPU and check the reported status.  The
// drain after a give-up always waits up to 1 s for the copies still in flight.
__device__ unsigned long long g_tma_wait_limit_ns = 1000000000ull;
constexpr uint64_t kDrainLimitNs = 1000000000ull;

int set_tma_wait_limit_ns(unsigned long long ns) {
    return cudaMemcpyToSymbol(g_tma_wait_limit_ns, &ns, sizeof(ns)) == cudaSuccess ? 0 : -1;
}

// Non-blocking probe of a phase.
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: false after limit_ns (or 2^26 polls) without the phase completing; with
// limit_ns = 0, false unless the phase has already completed (one non-blocking probe).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
    if (limit_ns == 0) return mbar_test_wait(bar, parity);
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    for (uint32_t it = 0; it < (1u << 26); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255u) == 0 && global_ns() - t0 > limit_ns) return false;
    }
    return false;
}
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1,
                                            int c2, int c3, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
        "r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int c0, int c1,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_addr(bar))
        : "memory");
}

__constant__ float g_tma_fs[4 * 9 + 3 * 8 + 4 * 8];
constexpr int TFS_UYY = 0, TFS_UY = 36, TFS_DWY = 60;

int upload_tma_tables(const double* fs_uyy, const double* fs_uy, const double* fs_dwy) {
    float f[92];
    for (int i = 0; i < 36; ++i) f[TFS_UYY + i] = (float)fs_uyy[i];
    for (int i = 0; i < 24; ++i) f[TFS_UY + i] = (float)fs_uy[i];
    for (int i = 0; i < 32; ++i) f[TFS_DWY + i] = (float)fs_dwy[i];
    return cudaMemcpyToSymbol(g_tma_fs, f, sizeof(f)) == cudaSuccess ? 0 : -1;
}

template <int R>
__device__ __forceinline__ float stag(int k) {
    if constexpr (R == 4) {
        return k == 0 ? float(1225.0 / 1024.0) : k == 1 ? float(-245.0 / 3072.0)
             : k == 2 ? float(49.0 / 5120.0) : float(-5.0 / 7168.0);
    } else {
        return k == 0 ? float(9.0 / 8.0) : float(-1.0 / 24.0);
    }
}
template <int R>
__device__ __forceinline__ float cent(int k) {
    if constexpr (R == 4) {
        return k == 0 ? float(-205.0 / 72.0) : k == 1 ? float(8.0 / 5.0) : k == 2 ? float(-1.0 / 5.0)
             : k == 3 ? float(8.0 / 315.0) : float(-1.0 / 560.0);
    } else {
        return k == 0 ? float(-5.0 / 2.0) : k == 1 ? float(4.0 / 3.0) : float(-1.0 / 12.0);
    }
}
// Stencil sums as balanced trees (short dependency chains for the issue slots):
// stag_tree = sum_k s_k d[k] over the R staggered differences, cent_tree = c_0 u +
// sum_k c_k p[k-1] over the R symmetric pair sums.
template <int R>
__device__ __forceinline__ float stag_tree(const float (&d)[R]) {
    if constexpr (R == 4)
        return fmaf(stag<4>(0), d[0], stag<4>(1) * d[1]) + fmaf(stag<4>(2), d[2], stag<4>(3) * d[3]);
    else
        return fmaf(stag<R>(0), d[0], stag<R>(1) * d[1]);
}
template <int R>
__device__ __forceinline__ float cent_tree(float u, const float (&p)[R]) {
    if constexpr (R == 4)
        return (fmaf(cent<4>(1), p[0], cent<4>(0) * u) + fmaf(cent<4>(3), p[2], cent<4>(2) * p[1])) +
               cent<4>(4) * p[3];
    else
        return fmaf(cent<R>(1), p[0], cent<R>(0) * u) + cent<R>(2) * p[1];
}

// Arithmetic on packed FP32 pairs (one instruction for both columns of a consumer thread; each
// component rounds exactly as the scalar operation does).
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 f2s(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2s(-1.f), a); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// beta at 2 d = k half cells from the first ghost line (zero beyond the layer).  Columns and
// rows past the grid edge (ragged tiles, never stored) give k <= 0; the unsigned test sends
// negative k to zero as well, so the table is never read outside its n entries.
__device__ __forceinline__ float btab_at(const float* t, int n, int k) {
    return (unsigned)k < (unsigned)n ? __ldg(t + k) : 0.f;
}

// Map of field box `kind` (0 u, 1 w_x, 2 w_y, 3 v, 4 four fields) for vector k.
__device__ __forceinline__ const CUtensorMap* map_of(const CUtensorMap* base, int k, int kind) {
    return base + (k == 0 ? 0 : 5) + kind;
}

// Problem of tile t: the last p with base[p] <= t (base: nprob + 1 prefix sums).
__device__ __forceinline__ int find_problem(const int* __restrict__ base, int nprob, int t) {
    int lo = 0, hi = nprob - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(base + mid) <= t) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The tile descriptor the producer hands to the consumers with a stage.
__device__ __forceinline__ void fill_tile_info(TileInfo& ti, const ProblemDev* P, const StageArgs& a, int x0,
                                               int y0) {
    ti.Y = a.y_out >= 0 ? (a.y_out == 0 ? (float*)P->state
                                        : (float*)P->work + (long long)(a.y_out - 1) * P->vec_stride)
                        : nullptr;
    ti.A = a.acc_out >= 0 ? (a.acc_out == 0 ? (float*)P->state
                                            : (float*)P->work + (long long)(a.acc_out - 1) * P->vec_stride)
                          : nullptr;
    ti.T = a.tape_vec > 0 ? (float*)P->work + (long long)(a.tape_vec - 1) * P->vec_stride +
                                (long long)a.tape_field * P->field_stride
                          : nullptr;
    ti.G = a.grad ? (float*)a.grad + (long long)P->shot * P->field_stride : nullptr;
    ti.fstr = P->field_stride;
    ti.x0 = x0;
    ti.y0 = y0;
    ti.nx = P->nx;
    ti.ny = P->ny;
    ti.pitch = P->pitch;
    ti.pml = P->pml;
    ti.fs = P->fs;
    ti.src_i = P->src_i;
    ti.src_j = P->src_j;
    ti.shot = P->shot;
    ti.btab = P->btab;
    ti.nbtab = P->nbtab;
    ti.xdamp = x0 - 8 < P->pml || x0 + BX + 8 > P->nx - P->pml;
    ti.beta0 = P->fbeta0;
    ti.inv_pml = P->finv_pml;
    ti.idx1 = P->finv_dx;
    ti.idx2 = P->finv_dx2;
}
// ... and the part that earlier kernels write.
__device__ __forceinline__ void fill_tile_scalars(TileInfo& ti, const ProblemDev* P, const StageArgs& a) {
    ti.sig = (a.src_slot >= 0 && P->has_src) ? (float)P->sigma[a.src_slot] : 0.f;
    ti.xs = a.x_scale_slot >= 0 ? (float)P->kry[a.x_scale_slot] : 1.f;
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory");
}

// The producer (one elected lane of the last warp): for each tile of this CTA, wait until
// its stage is free, resolve the tile's problem and descriptor, arm the stage's "full"
// barrier with the byte count and issue the TMA loads.  Returns the number of tiles issued.
// What no kernel writes (the first tile's descriptor, the tensor maps) is fetched before the wait
// for the pass before (pdl.cuh): with the shared memory cut to the stages in use (smem_in_use), a
// HORK stage on one shot takes 4.6 us instead of 5.0 on 301 x 201, 6.2 instead of 6.8 on 601 x 301,
// 9.3 instead of 9.8 on 1001 x 501.
template <int R, int BYv, int NSTv, int EPI, bool HASU, bool HASA = true>
__device__ __forceinline__ int tma_produce(const ProblemDev* __restrict__ probs, const int* __restrict__ tbase,
                                           int nprob, int ntiles, int mapset, const StageArgs& a, float* smem,
                                           uint64_t* full, uint64_t* empty, TileInfo* info, int* s_err,
                                           uint32_t bytes, uint64_t wait_lim) {
    using L = StageLayout<R, BYv, HASU, HASA>;
    const bool has_u = HASU && a.u >= 0, has_a = HASA && a.a >= 0;
    int issued = 0;
    int it = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
        const int s = it % NSTv;
        const uint32_t ph = (uint32_t)(it / NSTv) & 1u;
        // (the tile is resolved before the wait, so that a stage set free is refilled at once)
        const int pid = find_problem(tbase, nprob, tile);
        const ProblemDev* P = probs + pid;
        const CUtensorMap* maps = reinterpret_cast<const CUtensorMap*>(P->tmaps) + mapset * NMAP;
        const int tiles_x = (P->nx + BX - 1) / BX;
        const int lt = tile - __ldg(tbase + pid);
        const int x0 = (lt % tiles_x) * BX, y0 = (lt / tiles_x) * BYv;
        TileInfo ti;
        fill_tile_info(ti, P, a, x0, y0);
        if (it == 0) {
            for (int m = 0; m < 4; ++m) prefetch_map(map_of(maps, a.x, m));
            prefetch_map(maps + 10);
            if (has_u) prefetch_map(map_of(maps, a.u, 4));
            if (has_a) prefetch_map(map_of(maps, a.a, 4));
            pdl_wait();
        }
        fill_tile_scalars(ti, P, a);
        if (!mbar_wait(&empty[s], ph ^ 1u, wait_lim)) {
            *s_err = 1;
            break;
        }
        info[s] = ti;
        float* st = smem + (size_t)s * L::FLOATS;
        // the arrive below releases the tile info together with the copies
        mbar_expect_tx(&full[s], bytes);
        const int kx = a.x, cx = a.x == 0 ? 0 : a.x - 1;
        tma_load_4d(st + L::U_OFF, map_of(maps, kx, 0), x0 - TX, y0 - R, 0, cx, &full[s]);
        tma_load_4d(st + L::WX_OFF, map_of(maps, kx, 1), x0 - TX, y0, 2, cx, &full[s]);
        tma_load_4d(st + L::WY_OFF, map_of(maps, kx, 2), x0, y0 - R, 3, cx, &full[s]);
        if (EPI < 2) tma_load_4d(st + L::V_OFF, map_of(maps, kx, 3), x0, y0, 1, cx, &full[s]);
        if (EPI != 3) tma_load_2d(st + L::C2_OFF, maps + 10, x0, y0, &full[s]);
        if (has_u)
            tma_load_4d(st + L::PU_OFF, map_of(maps, a.u, 4), x0, y0, 0, a.u == 0 ? 0 : a.u - 1, &full[s]);
        if (has_a)
            tma_load_4d(st + L::PA_OFF, map_of(maps, a.a, 4), x0, y0, 0, a.a == 0 ? 0 : a.a - 1, &full[s]);
        issued = it + 1;
    }
    return issued;
}

// Byte count one stage receives (the "full" barrier's transaction count).
template <int R, int BYv, int EPI, bool HASU, bool HASA = true>
__device__ __forceinline__ uint32_t tma_stage_bytes(const StageArgs& a) {
    using L = StageLayout<R, BYv, HASU, HASA>;
    const bool has_u = HASU && a.u >= 0, has_a = HASA && a.a >= 0;
    // (the leap-frog step, EPI 2, does not read v; the gradient pass, EPI 3, neither v nor c^2)
    return (uint32_t)((L::BOX_FLOATS - (EPI >= 2 ? BYv * BX : 0) - (EPI == 3 ? BYv * BX : 0) +
                       (has_u ? 4 * BYv * BX : 0)) * 4) +
           (has_a ? 4 * BYv * BX * 4 : 0);
}

// After a pipeline wait gave up: the producer waits (bounded) for the last copy issued into
// every stage, so that no TMA write lands after the CTA exits, and the error word is set.
template <int NSTv>
__device__ __forceinline__ void tma_finish(int s_err, int issued, uint64_t* full, int* err) {
    const int tid = threadIdx.x;
    if (s_err) {
        if (issued > 0) {
            for (int it = issued - 1; it >= 0 && it >= issued - NSTv; --it)
                (void)mbar_wait(&full[it % NSTv], (uint32_t)(it / NSTv) & 1u, kDrainLimitNs);
        }
        if (tid == 0) atomicOr(err, 1);
    }
}

// ---------------------------------------------------------------- consumers
// Every consumer thread owns two adjacent columns (x, x + 1) of NR consecutive rows: the column
// pair of a staged row is one 8-byte shared load, and the arithmetic runs on packed FP32 pairs (one
// instruction for both columns).  The y taps of both columns slide in registers as pairs; the x
// taps of a row are the five pairs from x - 4 to x + 5, and the taps that straddle two pairs (odd
// offsets) are formed with scalar operations.  Per grid point this issues about a third of the
// shared loads of one column per thread and shares each tile's setup over twice the points.
// Every tile shape does the same arithmetic per point: the results do not depend on the variant
// the autotuner picks.  Rows of the free-surface band (Appendix A stencils, top tile only) take a
// scalar path per point.
// EPI 0: the general epilogue.  EPI 1: the steady-state form of the Faber and HORK passes, ck = 1
// and cau = cak = cax = 0:  Y = cu U + cx X + ch (H X + sigma),  ACC = ca A + cay Y.  EPI 2: one
// leap-frog step.  EPI 3: the gradient pass.
__device__ __forceinline__ float2 lds2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ void st2(float* p, float2 v, bool both) {
    if (both)
        *reinterpret_cast<float2*>(p) = v;
    else
        p[0] = v.x;
}

// One leap-frog step (Sec. 3.1) at a damped point: level n in registers, level n - 1 (u^{n-1},
// or d^n in field 1 in difference form, and w^{n-1}) from the A stage box at pa (fields plane
// floats apart); level n + 1 (u, w_x, w_y) goes to Y and, in difference form, d^{n+1} to field 1
// of A, which no thread of this step reads.
__device__ __forceinline__ void lf_point(const TileInfo& ti, const StageArgs& a, const float* pa, int plane, int ii,
                                         int jj, float uu, float c2v, float lap, float dws, float dux, float duy,
                                         float bxnv, float bxhv, float bynv, float byhv, float xwxv, float xwyv) {
    const float idx1 = ti.idx1, idx2 = ti.idx2;
    const float dt = (float)a.dt, bsum = bxnv + bynv;
    float rhs = -bxnv * bynv * uu + c2v * (lap * idx2 + dws * idx1);
    if (ii == ti.src_i && jj == ti.src_j) rhs += ti.sig;
    const long long o = (long long)jj * ti.pitch + ii;
    const long long fstr = ti.fstr;
    // fast (2-ulp) divisions: the step's own error is far larger
    float up;
    if (a.m == 2) {
        const float hb = 0.5f * bsum * dt;
        const float dn = __fdividef(pa[plane] * (1.f - hb) + dt * dt * rhs, 1.f + hb);
        ti.A[fstr + o] = dn;
        up = uu + dn;
    } else {
        const float um = pa[0];
        const float inv_dt2 = 1.f / (dt * dt), inv_2dt = 1.f / (2.f * dt);
        up = __fdividef((2.f * uu - um) * inv_dt2 + bsum * um * inv_2dt + rhs, inv_dt2 + bsum * inv_2dt);
    }
    float wxp = 0.f, wyp = 0.f;
    if (ii < ti.nx - 1) {
        const float gx = (bynv - bxhv) * dux * idx1, wm = pa[2 * plane];
        wxp = a.m != 1 ? __fdividef((1.f - bxhv * dt) * wm + 2.f * dt * gx, 1.f + bxhv * dt)
                       : wm + 2.f * dt * (-bxhv * xwxv + gx);
    }
    if (jj < ti.ny - 1) {
        const float gy = (bxnv - byhv) * duy * idx1, wm = pa[3 * plane];
        wyp = a.m != 1 ? __fdividef((1.f - byhv * dt) * wm + 2.f * dt * gy, 1.f + byhv * dt)
                       : wm + 2.f * dt * (-byhv * xwyv + gy);
    }
    ti.Y[o] = up;
    ti.Y[2 * fstr + o] = wxp;
    ti.Y[3 * fstr + o] = wyp;
}

// One point (tile column tc, tile row lr) from shared memory with scalar formulas, free-surface
// rows included, and its epilogue.
template <int R, int BYv, int EPI, bool HASU, bool HASA>
__device__ __forceinline__ void tma_point_scalar(const float* st, const TileInfo& ti, const StageArgs& a, int tc,
                                             int lr, bool has_u, bool has_a) {
    using L = StageLayout<R, BYv, HASU, HASA>;
    const int nx = ti.nx, ny = ti.ny;
    const int i = ti.x0 + tc, j = ti.y0 + lr;
    if (i >= nx || j >= ny) return;
    const bool fs = ti.fs != 0;
    const int cs = tc + TX;
    const float* su = st + L::U_OFF;
    const float* swy = st + L::WY_OFF;
    const float* urow = su + (lr + R) * L::SW + cs;
    const float* wxrow = st + L::WX_OFF + lr * L::SW + cs;
    auto ucolv = [&](int q) { return su[(lr + q) * L::SW + cs]; };   // staged row lr + q
    auto wcolv = [&](int q) { return swy[(lr + q) * BX + tc]; };
    float px[R], dx[R], dw[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        px[k] = urow[k + 1] + urow[-k - 1];
        dx[k] = urow[1 + k] - urow[-k];
        dw[k] = wxrow[k] - wxrow[-1 - k];
    }
    const float uc = urow[0];
    const float uxx = cent_tree<R>(uc, px);
    const float dux = stag_tree<R>(dx);
    const float dwx = stag_tree<R>(dw);
    float uyy, duy, dwy;
    if (fs && j < 4) {
        uyy = 0.f;
#pragma unroll
        for (int q = 0; q < 9; ++q) uyy += g_tma_fs[TFS_UYY + j * 9 + q] * su[(q + R) * L::SW + cs];
        dwy = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) dwy += g_tma_fs[TFS_DWY + j * 8 + q] * swy[(q + R) * BX + tc];
    } else {
        float py[R], dwv[R];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            py[k] = ucolv(R + k + 1) + ucolv(R - k - 1);
            dwv[k] = wcolv(R - 1 - k) - wcolv(R + k);
        }
        uyy = cent_tree<R>(uc, py);
        dwy = stag_tree<R>(dwv);
    }
    if (fs && j < 3) {
        duy = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) duy += g_tma_fs[TFS_UY + j * 8 + q] * su[(q + R) * L::SW + cs];
    } else {
        float dy[R];
#pragma unroll
        for (int k = 0; k < R; ++k) dy[k] = ucolv(R - k) - ucolv(R + 1 + k);
        duy = stag_tree<R>(dy);
    }
    const float* btab = ti.btab;
    const int nbt = ti.nbtab;
    const float bxn = btab_at(btab, nbt, 2 * min(i + 1, nx - i));
    const float bxh = btab_at(btab, nbt, min(2 * i + 3, 2 * (nx - i) - 1));
    const float byn = btab_at(btab, nbt, 2 * (fs ? ny - j : min(j + 1, ny - j)));
    const float byh = btab_at(btab, nbt, fs ? 2 * (ny - j) - 1 : min(2 * j + 3, 2 * (ny - j) - 1));
    const int pt = lr * BX + tc;
    const float* sv = st + L::V_OFF;
    const float* sc2 = st + L::C2_OFF;
    const float* spu = st + L::PU_OFF;
    const float* spa = st + L::PA_OFF;
    if constexpr (EPI == 3) {
        float* G = (float*)a.grad + (long long)ti.shot * ti.fstr;
        G[(long long)j * ti.pitch + i] +=
            (float)a.gscale * spa[BYv * BX + pt] * ((uxx + uyy) * ti.idx2 + (dwx + dwy) * ti.idx1);
        return;
    }
    if constexpr (EPI == 2) {
        lf_point(ti, a, spa + pt, BYv * BX, i, j, uc, sc2[pt], uxx + uyy, dwx + dwy, dux, duy, bxn, bxh, byn,
                 byh, wxrow[0], wcolv(R));
        return;
    }
    const float idx1 = ti.idx1, idx2 = ti.idx2;
    if (ti.T) ti.T[(long long)j * ti.pitch + i] = (uxx + uyy) * idx2 + (dwx + dwy) * idx1;
    const float xu = uc, xv = sv[pt], xwx = wxrow[0], xwy = wcolv(R);
    float hv = -bxn * byn * xu + sc2[pt] * ((uxx + uyy) * idx2 + (dwx + dwy) * idx1) - (bxn + byn) * xv;
    if (i == ti.src_i && j == ti.src_j) hv += ti.sig;
    const float hwx = (i < nx - 1) ? (byn - bxh) * dux * idx1 - bxh * xwx : 0.f;
    const float hwy = (j < ny - 1) ? (bxn - byh) * duy * idx1 - byh * xwy : 0.f;
    const float xf[4] = {xu, xv, xwx, xwy};
    const float hf[4] = {xv, hv, hwx, hwy};
    const float chx = a.fch * ti.xs;
    const long long o = (long long)j * ti.pitch + i;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        const bool pad = (f == 2 && i >= nx - 1) || (f == 3 && j >= ny - 1);
        const float uval = has_u ? spu[f * BYv * BX + pt] : 0.f;
        const float aval = has_a ? spa[f * BYv * BX + pt] : 0.f;
        const float kf = fmaf(a.fcx, xf[f], chx * hf[f]);
        if constexpr (EPI == 1) {
            const float yf = pad ? 0.f : (has_u ? fmaf(a.fcu, uval, kf) : kf);
            if (ti.Y) ti.Y[f * ti.fstr + o] = yf;
            if (ti.A) ti.A[f * ti.fstr + o] = has_a ? fmaf(a.fcay, yf, a.fca * aval) : a.fcay * yf;
        } else {
            const float yf = pad ? 0.f : (a.fcu * uval + a.fck * kf);
            if (ti.Y) ti.Y[f * ti.fstr + o] = yf;
            if (ti.A)
                ti.A[f * ti.fstr + o] =
                    pad ? 0.f : (a.fca * aval + a.fcau * uval + a.fcak * kf + a.fcay * yf + a.fcax * xf[f]);
        }
    }
}

template <int R, int BYv, int NW, int NSTv, int EPI, bool HASU, bool HASA>
__global__ void __launch_bounds__(NW * 32 + 32, 1)
stage_tma_x2_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ tbase, int nprob,
                    int ntiles, int mapset, StageArgs a, int* err) {
    static_assert(EPI <= 3, "EPI 0 / 1: integrator passes, 2: leap-frog step, 3: gradient pass");
    using L = StageLayout<R, BYv, HASU, HASA>;
    constexpr int CPR = BX / 2;                 // consumer threads per tile row
    constexpr int TPR = NW * 32 / CPR;          // thread rows
    constexpr int NR = BYv / TPR;               // consecutive rows per consumer thread
    static_assert(NR * TPR == BYv && NR >= 1, "tile rows must split evenly over threads");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    float* smem = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[NSTv];
    __shared__ __align__(8) uint64_t empty[NSTv];
    __shared__ TileInfo info[NSTv];
    __shared__ int s_err;

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const uint64_t wait_lim = g_tma_wait_limit_ns;
    if (tid == 0) {
        for (int s = 0; s < NSTv; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], NW);
        }
        s_err = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_trigger();
    if (warp != NW) pdl_wait();     // (the producer's own wait comes after the first tile is resolved)
    const bool has_u = HASU && a.u >= 0, has_a = HASA && a.a >= 0;
    int issued = 0;
    if (warp == NW) {
        if (lane == 0)
            issued = tma_produce<R, BYv, NSTv, EPI, HASU, HASA>(
                probs, tbase, nprob, ntiles, mapset, a, smem, full, empty, info, &s_err,
                tma_stage_bytes<R, BYv, EPI, HASU, HASA>(a), wait_lim);
    } else {
        const int tx2 = tid % CPR, ty = tid / CPR;
        const int c0 = 2 * tx2;                 // first of the two tile columns
        const int cs = c0 + TX;                 // its staged column (even: 8-byte aligned)
        const int r0 = NR * ty;                 // first tile row of this thread
        const float2 cx2 = f2s(a.fcx), cu2 = f2s(a.fcu), ck2 = f2s(a.fck), ca2 = f2s(a.fca);
        const float2 cay2 = f2s(a.fcay), cau2 = f2s(a.fcau), cak2 = f2s(a.fcak), cax2 = f2s(a.fcax);
        int it = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
            const int s = it % NSTv;
            const uint32_t ph = (uint32_t)(it / NSTv) & 1u;
            if (!mbar_wait(&full[s], ph, wait_lim)) {
                s_err = 1;
                break;
            }
            const TileInfo ti = load_info(&info[s]);
            const float* st = smem + (size_t)s * L::FLOATS;
            const int nx = ti.nx, ny = ti.ny;
            const int i0 = ti.x0 + c0;
            const int jt = ti.y0 + r0;
            if (i0 < nx && jt < ny) {
                if (ti.fs != 0 && jt < 4) {
                    // free-surface band: one point at a time
#pragma unroll 1
                    for (int r = 0; r < NR; ++r) {
                        tma_point_scalar<R, BYv, EPI, HASU, HASA>(st, ti, a, c0, r0 + r, has_u, has_a);
                        tma_point_scalar<R, BYv, EPI, HASU, HASA>(st, ti, a, c0 + 1, r0 + r, has_u, has_a);
                    }
                } else {
                    const float* su = st + L::U_OFF;
                    const float* swx = st + L::WX_OFF;
                    const float* swy = st + L::WY_OFF;
                    const float* sv = st + L::V_OFF;
                    const float* sc2 = st + L::C2_OFF;
                    const float* spu = st + L::PU_OFF;
                    const float* spa = st + L::PA_OFF;
                    const bool fs = ti.fs != 0;
                    const bool in1 = i0 + 1 < nx;
                    float2 ucol[NR + 2 * R], wcol[NR + 2 * R - 1];
#pragma unroll
                    for (int q = 0; q < NR + 2 * R; ++q) ucol[q] = lds2(su + (r0 + q) * L::SW + cs);
#pragma unroll
                    for (int q = 0; q < NR + 2 * R - 1; ++q) wcol[q] = lds2(swy + (r0 + q) * BX + c0);
                    const float* btab = ti.btab;
                    const int nbt = ti.nbtab;
                    // Where nothing damps this thread's points, the w rows of H are zero and the v
                    // row has no damping term: no look-ups, no half-point differences of u (the
                    // results are the same to the bit; about a fifth of the instructions).
                    const bool damped = ti.xdamp || jt + NR > ny - ti.pml || (!fs && jt < ti.pml);
                    float2 bxn = f2s(0.f), bxh = f2s(0.f), nbxh = f2s(0.f);
                    if (damped) {
                        bxn = f2(btab_at(btab, nbt, 2 * min(i0 + 1, nx - i0)),
                                 btab_at(btab, nbt, 2 * min(i0 + 2, nx - i0 - 1)));
                        bxh = f2(btab_at(btab, nbt, min(2 * i0 + 3, 2 * (nx - i0) - 1)),
                                 btab_at(btab, nbt, min(2 * i0 + 5, 2 * (nx - i0) - 3)));
                        nbxh = f2(-bxh.x, -bxh.y);
                    }
                    const bool wx0in = i0 < nx - 1, wx1in = i0 + 1 < nx - 1;
                    const float2 idx1 = f2s(ti.idx1), idx2 = f2s(ti.idx2);
                    const float chx = a.fch * ti.xs;
                    const float2 chx2 = f2s(chx);
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        const int lr = r0 + r, j = jt + r;
                        if (j >= ny) break;
                        // x taps: u and w_x at tile columns c0 - 4 .. c0 + 5 of this row
                        const float* urow = su + (lr + R) * L::SW + cs;
                        const float* wxr = swx + lr * L::SW + cs;
                        const float2 up[5] = {lds2(urow - 4), lds2(urow - 2), ucol[r + R], lds2(urow + 2),
                                              lds2(urow + 4)};
                        const float2 wp[5] = {lds2(wxr - 4), lds2(wxr - 2), lds2(wxr), lds2(wxr + 2),
                                              lds2(wxr + 4)};
                        // scalar tap at column offset d (-4 .. 5) from the first column
                        auto uo = [&](int d) { return ((d + 4) & 1) ? up[(d + 4) >> 1].y : up[(d + 4) >> 1].x; };
                        auto wo = [&](int d) { return ((d + 4) & 1) ? wp[(d + 4) >> 1].y : wp[(d + 4) >> 1].x; };
                        const float2 uc = ucol[r + R];
                        float2 lap = mul2(f2s(2.f * cent<R>(0)), uc);
                        float2 dux = f2s(0.f), duy = f2s(0.f), dw = f2s(0.f);
                        float byn = 0.f, byh = 0.f;
                        if (EPI != 3 && damped) {
                            byn = btab_at(btab, nbt, 2 * (fs ? ny - j : min(j + 1, ny - j)));
                            byh = btab_at(btab, nbt, fs ? 2 * (ny - j) - 1 : min(2 * j + 3, 2 * (ny - j) - 1));
                            // staggered differences: d_x u at x + 1/2, d_y u at y + 1/2
#pragma unroll
                            for (int k = 0; k < R; ++k) {
                                const float2 dxu = f2(uo(1 + k) - uo(-k), uo(2 + k) - uo(1 - k));
                                dux = fma2(f2s(stag<R>(k)), dxu, dux);
                                duy = fma2(f2s(stag<R>(k)), sub2(ucol[r + R - k], ucol[r + R + 1 + k]), duy);
                            }
                        }
#pragma unroll
                        for (int k = 0; k < R; ++k) {
                            // Laplacian: x and y pair sums at distance k + 1
                            const int kk = k + 1;
                            const float2 sx = (kk & 1) ? f2(uo(kk) + uo(-kk), uo(kk + 1) + uo(1 - kk))
                                                       : add2(up[(kk + 4) >> 1], up[(4 - kk) >> 1]);
                            const float2 sy = add2(ucol[r + R + kk], ucol[r + R - kk]);
                            lap = fma2(f2s(cent<R>(kk)), add2(sx, sy), lap);
                            // the divergence of w at the node
                            const float2 dxw = f2(wo(k) - wo(-1 - k), wo(1 + k) - wo(-k));
                            const float2 dyw = sub2(wcol[r + R - 1 - k], wcol[r + R + k]);
                            dw = fma2(f2s(stag<R>(k)), add2(dxw, dyw), dw);
                        }
                        const int pt = lr * BX + c0;
                        if constexpr (EPI == 3) {
                            // FWI gradient pass: grad += gscale q_v (L u + D w) of X (m = c^2);
                            // q's fields ride in the A box
                            float* G = (float*)a.grad + (long long)ti.shot * ti.fstr +
                                       (long long)j * ti.pitch + i0;
                            const float2 qv = lds2(spa + BYv * BX + pt);
                            const float2 gv = mul2(mul2(f2s((float)a.gscale), qv),
                                                   fma2(lap, f2s(ti.idx2), mul2(dw, f2s(ti.idx1))));
                            if (in1) {
                                float2 g0 = *reinterpret_cast<float2*>(G);
                                *reinterpret_cast<float2*>(G) = add2(g0, gv);
                            } else {
                                G[0] += gv.x;
                            }
                            continue;
                        }
                        if constexpr (EPI == 2) {
                            // one leap-frog step per column of the pair
                            const float2 c2l = lds2(sc2 + pt);
                            if (!damped) {
                                // no damping: w keeps its level n-1 values, u needs no division
                                const float* pa = spa + pt;
                                const long long o = (long long)j * ti.pitch + i0;
                                const float2 dt2 = f2s((float)a.dt * (float)a.dt);
                                float2 rhs = mul2(c2l, fma2(lap, idx2, mul2(dw, idx1)));
                                if (j == ti.src_j) {
                                    if (i0 == ti.src_i) rhs.x += ti.sig;
                                    if (i0 + 1 == ti.src_i) rhs.y += ti.sig;
                                }
                                float2 up;
                                if (a.m == 2) {
                                    const float2 dn = fma2(dt2, rhs, lds2(pa + BYv * BX));
                                    st2(ti.A + ti.fstr + o, dn, in1);
                                    up = add2(uc, dn);
                                } else {
                                    up = fma2(dt2, rhs, fma2(f2s(2.f), uc, mul2(f2s(-1.f), lds2(pa))));
                                }
                                float2 wxp = lds2(pa + 2 * BYv * BX), wyp = lds2(pa + 3 * BYv * BX);
                                if (!wx0in) wxp.x = 0.f;
                                if (!wx1in) wxp.y = 0.f;
                                if (j >= ny - 1) wyp = f2s(0.f);
                                st2(ti.Y + o, up, in1);
                                st2(ti.Y + 2 * ti.fstr + o, wxp, in1);
                                st2(ti.Y + 3 * ti.fstr + o, wyp, in1);
                                continue;
                            }
                            lf_point(ti, a, spa + pt, BYv * BX, i0, j, uc.x, c2l.x, lap.x, dw.x, dux.x, duy.x,
                                     bxn.x, bxh.x, byn, byh, wp[2].x, wcol[r + R].x);
                            if (in1)
                                lf_point(ti, a, spa + pt + 1, BYv * BX, i0 + 1, j, uc.y, c2l.y, lap.y, dw.y, dux.y,
                                         duy.y, bxn.y, bxh.y, byn, byh, wp[2].y, wcol[r + R].y);
                            continue;
                        }
                        const float2 xv = lds2(sv + pt), c2 = lds2(sc2 + pt);
                        const float2 xwx = wp[2], xwy = wcol[r + R];
                        // H v = -bx by u + c^2 (lap u / dx^2 + div w / dx) - (bx + by) v
                        const float2 force = fma2(lap, idx2, mul2(dw, idx1));
                        // tape pass of an adjoint step: L u + D w, the gradient's factor of this vector
                        if (ti.T) st2(ti.T + (long long)j * ti.pitch + i0, force, in1);
                        const bool wyin = j < ny - 1;
                        float2 hv, hwx = f2s(0.f), hwy = f2s(0.f);
                        if (damped) {
                            const float2 t = fma2(mul2(bxn, f2s(-byn)), uc, mul2(sub2(f2s(-byn), bxn), xv));
                            hv = fma2(c2, force, t);
                            hwx = fma2(nbxh, xwx, mul2(mul2(sub2(f2s(byn), bxh), dux), idx1));
                            if (!wx0in) hwx.x = 0.f;
                            if (!wx1in) hwx.y = 0.f;
                            if (wyin) hwy = fma2(f2s(-byh), xwy, mul2(mul2(sub2(bxn, f2s(byh)), duy), idx1));
                        } else {
                            hv = mul2(c2, force);
                        }
                        if (j == ti.src_j) {
                            if (i0 == ti.src_i) hv.x += ti.sig;
                            if (i0 + 1 == ti.src_i) hv.y += ti.sig;
                        }
                        const float2 xf[4] = {uc, xv, xwx, xwy};
                        const float2 hf[4] = {xv, hv, hwx, hwy};
                        const long long o = (long long)j * ti.pitch + i0;
#pragma unroll
                        for (int f = 0; f < 4; ++f) {
                            const float2 uval = has_u ? lds2(spu + f * BYv * BX + pt) : f2s(0.f);
                            const float2 aval = has_a ? lds2(spa + f * BYv * BX + pt) : f2s(0.f);
                            const float2 kf = fma2(cx2, xf[f], mul2(chx2, hf[f]));
                            float2 yf, af;
                            if constexpr (EPI == 1) {
                                yf = has_u ? fma2(cu2, uval, kf) : kf;
                            } else {
                                yf = fma2(cu2, uval, mul2(ck2, kf));
                            }
                            if (f == 2) {
                                if (!wx0in) yf.x = 0.f;
                                if (!wx1in) yf.y = 0.f;
                            }
                            if (f == 3 && !wyin) yf = f2s(0.f);
                            if constexpr (EPI == 1) {
                                af = has_a ? fma2(cay2, yf, mul2(ca2, aval)) : mul2(cay2, yf);
                            } else {
                                af = fma2(cax2, xf[f],
                                          fma2(cay2, yf, fma2(cak2, kf, fma2(cau2, uval, mul2(ca2, aval)))));
                                if (f == 2) {
                                    if (!wx0in) af.x = 0.f;
                                    if (!wx1in) af.y = 0.f;
                                }
                                if (f == 3 && !wyin) af = f2s(0.f);
                            }
                            if (ti.Y) st2(ti.Y + f * ti.fstr + o, yf, in1);
                            if (ti.A) st2(ti.A + f * ti.fstr + o, af, in1);
                        }
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[s]);
        }
    }
    __syncthreads();
    tma_finish<NSTv>(s_err, issued, full, err);
}

// ---------------------------------------------------------------- transposed pass
// H^T y (the adjoint's passes) with the column-pair consumers.  For y = (y_u, y_v, y_wx,
// y_wy):
//   (H^T y)_u  = -bx by y_v + L (c^2 y_v) - D_x(z_x) - D_y(z_y)      (L symmetric in the interior)
//   (H^T y)_v  = y_u - (bx + by) y_v
//   (H^T y)_wx = -d_x^+(c^2 y_v) - bx^h y_wx                          at (i+1/2, j)
//   (H^T y)_wy = -d_y^+(c^2 y_v) - by^h y_wy                          at (i, j+1/2)
// with z_x = (by - bx^h) y_wx at the half columns and z_y = (bx - by^h) y_wy at the half rows:
// the transposes of the forward's staggered derivatives are the negated staggered
// derivatives of the other grid (zero extension keeps that exact at the edges).  The stage
// carries y_v and c^2 with the 2D halo (their product is formed from shared memory), y_wx
// with the x halo, y_wy with the y halo, y_u and the U / A operands.  The rows whose
// transposed stencils meet the free-surface rows of Appendix A (rows 0..8: the columns of
// those rows) take a scalar path per point that adds the tables' columns.
template <int R, int BYv, bool HASU, bool HASA>
struct TLayout {
    static constexpr int up32(int v) { return (v + 31) / 32 * 32; }
    static constexpr int SH = BYv + 2 * R;
    static constexpr int SW = BX + 2 * TX;
    static constexpr int ZV_OFF = 0;                                 // y_v    SH x SW
    static constexpr int C2_OFF = up32(ZV_OFF + SH * SW);            // c^2    SH x SW
    static constexpr int WX_OFF = up32(C2_OFF + SH * SW);            // y_wx   BYv x SW
    static constexpr int WY_OFF = up32(WX_OFF + BYv * SW);           // y_wy   SH x BX
    static constexpr int YU_OFF = WY_OFF + SH * BX;                  // y_u    BYv x BX
    static constexpr int PU_OFF = YU_OFF + BYv * BX;                 // U      4 x BYv x BX
    static constexpr int PA_OFF = PU_OFF + (HASU ? 4 * BYv * BX : 0);   // A   4 x BYv x BX
    static constexpr int FLOATS = PA_OFF + (HASA ? 4 * BYv * BX : 0);
    static constexpr int BOX_FLOATS = 2 * SH * SW + BYv * SW + SH * BX + BYv * BX;
    static constexpr int BYTES = FLOATS * 4;
    static_assert((C2_OFF * 4) % 128 == 0 && (WX_OFF * 4) % 128 == 0 && (WY_OFF * 4) % 128 == 0 &&
                      (YU_OFF * 4) % 128 == 0 && (PU_OFF * 4) % 128 == 0 && (PA_OFF * 4) % 128 == 0 &&
                      BYTES % 128 == 0,
                  "TMA destinations must be 128-byte aligned");
};

template <int R, int BYv, int NSTv, bool HASU, bool HASA>
__device__ __forceinline__ int tma_produce_t(const ProblemDev* __restrict__ probs, const int* __restrict__ tbase,
                                             int nprob, int ntiles, int mapset, const StageArgs& a, float* smem,
                                             uint64_t* full, uint64_t* empty, TileInfo* info, int* s_err,
                                             uint64_t wait_lim) {
    using L = TLayout<R, BYv, HASU, HASA>;
    const bool has_u = HASU && a.u >= 0, has_a = HASA && a.a >= 0;
    const uint32_t bytes = (uint32_t)(L::BOX_FLOATS + (has_u ? 4 * BYv * BX : 0) + (has_a ? 4 * BYv * BX : 0)) * 4u;
    int issued = 0;
    int it = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
        const int s = it % NSTv;
        const uint32_t ph = (uint32_t)(it / NSTv) & 1u;
        // (the tile is resolved before the wait, so that a stage set free is refilled at once)
        const int pid = find_problem(tbase, nprob, tile);
        const ProblemDev* P = probs + pid;
        const CUtensorMap* maps = reinterpret_cast<const CUtensorMap*>(P->tmaps) + mapset * NMAP;
        const int tiles_x = (P->nx + BX - 1) / BX;
        const int lt = tile - __ldg(tbase + pid);
        const int x0 = (lt % tiles_x) * BX, y0 = (lt / tiles_x) * BYv;
        TileInfo ti;
        fill_tile_info(ti, P, a, x0, y0);
        if (it == 0) {
            for (int m = 0; m < 4; ++m) prefetch_map(map_of(maps, a.x, m));
            prefetch_map(maps + 11);
            if (has_u) prefetch_map(map_of(maps, a.u, 4));
            if (has_a) prefetch_map(map_of(maps, a.a, 4));
            pdl_wait();
        }
        fill_tile_scalars(ti, P, a);
        if (!mbar_wait(&empty[s], ph ^ 1u, wait_lim)) {
            *s_err = 1;
            break;
        }
        info[s] = ti;
        float* st = smem + (size_t)s * L::FLOATS;
        mbar_expect_tx(&full[s], bytes);
        const int kx = a.x, cx = a.x == 0 ? 0 : a.x - 1;
        tma_load_4d(st + L::ZV_OFF, map_of(maps, kx, 0), x0 - TX, y0 - R, 1, cx, &full[s]);   // y_v, 2D halo
        tma_load_2d(st + L::C2_OFF, maps + 11, x0 - TX, y0 - R, &full[s]);                   // c^2, 2D halo
        tma_load_4d(st + L::WX_OFF, map_of(maps, kx, 1), x0 - TX, y0, 2, cx, &full[s]);
        tma_load_4d(st + L::WY_OFF, map_of(maps, kx, 2), x0, y0 - R, 3, cx, &full[s]);
        tma_load_4d(st + L::YU_OFF, map_of(maps, kx, 3), x0, y0, 0, cx, &full[s]);           // y_u
        if (has_u)
            tma_load_4d(st + L::PU_OFF, map_of(maps, a.u, 4), x0, y0, 0, a.u == 0 ? 0 : a.u - 1, &full[s]);
        if (has_a)
            tma_load_4d(st + L::PA_OFF, map_of(maps, a.a, 4), x0, y0, 0, a.a == 0 ? 0 : a.a - 1, &full[s]);
        issued = it + 1;
    }
    return issued;
}

// The general epilogue (StageArgs) of one point: K = cx X + ch xs HX, Y = cu U + ck K,
// ACC = ca A + cau U + cak K + cay Y + cax X, pads of w_x / w_y zero.
__device__ __forceinline__ void tma_epilogue_point(const TileInfo& ti, const StageArgs& a, long long o, const float* xf,
                                                   const float* hf, const float* uv, const float* av, bool padx,
                                                   bool pady) {
    const float chx = a.fch * ti.xs;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        const bool pad = (f == 2 && padx) || (f == 3 && pady);
        const float kf = fmaf(a.fcx, xf[f], chx * hf[f]);
        const float yf = pad ? 0.f : (a.fcu * uv[f] + a.fck * kf);
        if (ti.Y) ti.Y[f * ti.fstr + o] = yf;
        if (ti.A)
            ti.A[f * ti.fstr + o] =
                pad ? 0.f : (a.fca * av[f] + a.fcau * uv[f] + a.fcak * kf + a.fcay * yf + a.fcax * xf[f]);
    }
}

// One transposed point from shared memory with the free-surface columns (rows 0..8 of the
// top tile), following the row structure of the forward operator.
template <int R, int BYv, bool HASU, bool HASA>
__device__ __forceinline__ void tma_point_scalar_t(const float* st, const TileInfo& ti, const StageArgs& a, int tc,
                                                   int lr, bool has_u, bool has_a) {
    using L = TLayout<R, BYv, HASU, HASA>;
    const int nx = ti.nx, ny = ti.ny;
    const int i = ti.x0 + tc, j = ti.y0 + lr;
    if (i >= nx || j >= ny) return;
    const bool fs = ti.fs != 0;
    const int cs = tc + TX;
    const float* btab = ti.btab;
    const int nbt = ti.nbtab;
    const float* zv_ = st + L::ZV_OFF;
    const float* c2_ = st + L::C2_OFF;
    const float* wx_ = st + L::WX_OFF;
    const float* wy_ = st + L::WY_OFF;
    // z_v at staged row q (grid row y0 + q - R), tile column tc + d
    auto zv = [&](int q, int d) { return zv_[q * L::SW + cs + d] * c2_[q * L::SW + cs + d]; };
    const float byn = btab_at(btab, nbt, 2 * (fs ? ny - j : min(j + 1, ny - j)));
    const float bxn = btab_at(btab, nbt, 2 * min(i + 1, nx - i));
    const float bxh = btab_at(btab, nbt, min(2 * i + 3, 2 * (nx - i) - 1));
    const float byh = btab_at(btab, nbt, fs ? 2 * (ny - j) - 1 : min(2 * j + 3, 2 * (ny - j) - 1));
    // z_x at half column i + d + 1/2 of this row, z_y at half row h of this column
    auto zx = [&](int d) {
        const int p = i + d;
        const float bh = btab_at(btab, nbt, min(2 * p + 3, 2 * (nx - p) - 1));
        return (byn - bh) * wx_[lr * L::SW + cs + d];
    };
    auto zy = [&](int h) {
        const float bh = btab_at(btab, nbt, fs ? 2 * (ny - h) - 1 : min(2 * h + 3, 2 * (ny - h) - 1));
        return (bxn - bh) * wy_[(h - ti.y0 + R) * BX + tc];
    };
    const int q0 = lr + R;   // staged row of j
    float lxx = cent<R>(0) * zv(q0, 0);
#pragma unroll
    for (int k = 1; k <= R; ++k) lxx += cent<R>(k) * (zv(q0, k) + zv(q0, -k));
    float lyy = 0.f;
    const int rfs = fs ? 4 : 0;
#pragma unroll
    for (int k = -R; k <= R; ++k) {
        const int r = j + k;
        if (r >= rfs && r < ny) lyy += cent<R>(k < 0 ? -k : k) * zv(q0 + k, 0);
    }
    if (fs && j <= 8) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (r < ny) lyy += g_tma_fs[TFS_UYY + r * 9 + j] * zv(r - ti.y0 + R, 0);
    }
    float gxt = 0.f;
#pragma unroll
    for (int k = 0; k < R; ++k) gxt += stag<R>(k) * (zx(-1 - k) - zx(k));
    float gyt = 0.f;
    const int hfs = fs ? 3 : 0;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int h1 = j + k, h2 = j - 1 - k;
        if (h1 >= hfs && h1 < ny - 1) gyt += stag<R>(k) * zy(h1);
        if (h2 >= hfs && h2 >= 0) gyt -= stag<R>(k) * zy(h2);
    }
    if (fs && j <= 7) {
#pragma unroll
        for (int h = 0; h < 3; ++h)
            if (h < ny - 1) gyt += g_tma_fs[TFS_UY + h * 8 + j] * zy(h);
    }
    float dxt = 0.f;
#pragma unroll
    for (int k = 0; k < R; ++k) dxt += stag<R>(k) * (zv(q0, -k) - zv(q0, 1 + k));
    float dyt = 0.f;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int r1 = j + 1 + k, r2 = j - k;
        if (r1 >= rfs && r1 < ny) dyt += stag<R>(k) * zv(q0 + 1 + k, 0);
        if (r2 >= rfs && r2 >= 0) dyt -= stag<R>(k) * zv(q0 - k, 0);
    }
    if (fs && j <= 7) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (r < ny) dyt += g_tma_fs[TFS_DWY + r * 8 + j] * zv(r - ti.y0 + R, 0);
    }
    const int pt = lr * BX + tc;
    const float yu = st[L::YU_OFF + pt], yv = zv_[q0 * L::SW + cs];
    const float ywx = (i < nx - 1) ? wx_[lr * L::SW + cs] : 0.f;
    const float ywy = (j < ny - 1) ? wy_[q0 * BX + tc] : 0.f;
    const float idx1 = ti.idx1, idx2 = ti.idx2;
    const float xf[4] = {yu, yv, ywx, ywy};
    const float hf[4] = {-bxn * byn * yv + (lxx + lyy) * idx2 + (gxt + gyt) * idx1, yu - (bxn + byn) * yv,
                         (i < nx - 1) ? dxt * idx1 - bxh * ywx : 0.f, (j < ny - 1) ? dyt * idx1 - byh * ywy : 0.f};
    float uv[4], av[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        uv[f] = has_u ? st[L::PU_OFF + f * BYv * BX + pt] : 0.f;
        av[f] = has_a ? st[L::PA_OFF + f * BYv * BX + pt] : 0.f;
    }
    const long long o = (long long)j * ti.pitch + i;
    if (ti.T) ti.G[o] += (float)a.gscale * yv * ti.T[o];
    tma_epilogue_point(ti, a, o, xf, hf, uv, av, i >= nx - 1, j >= ny - 1);
}

template <int R, int BYv, int NW, int NSTv, bool HASU, bool HASA>
__global__ void __launch_bounds__(NW * 32 + 32, 1)
stage_tma_t_kernel(const ProblemDev* __restrict__ probs, const int* __restrict__ tbase, int nprob, int ntiles,
                   int mapset, StageArgs a, int* err) {
    using L = TLayout<R, BYv, HASU, HASA>;
    constexpr int CPR = BX / 2;
    constexpr int TPR = NW * 32 / CPR;
    constexpr int NR = BYv / TPR;
    static_assert(NR * TPR == BYv && NR >= 1, "tile rows must split evenly over threads");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    float* smem = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[NSTv];
    __shared__ __align__(8) uint64_t empty[NSTv];
    __shared__ TileInfo info[NSTv];
    __shared__ int s_err;
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const uint64_t wait_lim = g_tma_wait_limit_ns;
    if (tid == 0) {
        for (int s = 0; s < NSTv; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], NW);
        }
        s_err = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_trigger();
    if (warp != NW) pdl_wait();     // (the producer's own wait comes after the first tile is resolved)
    const bool has_u = HASU && a.u >= 0, has_a = HASA && a.a >= 0;
    int issued = 0;
    if (warp == NW) {
        if (lane == 0)
            issued = tma_produce_t<R, BYv, NSTv, HASU, HASA>(probs, tbase, nprob, ntiles, mapset, a, smem, full,
                                                             empty, info, &s_err, wait_lim);
    } else {
        const int tx2 = tid % CPR, ty = tid / CPR;
        const int c0 = 2 * tx2, cs = c0 + TX, r0 = NR * ty;
        const float2 cx2 = f2s(a.fcx), cu2 = f2s(a.fcu), ck2 = f2s(a.fck), ca2 = f2s(a.fca);
        const float2 cay2 = f2s(a.fcay), cau2 = f2s(a.fcau), cak2 = f2s(a.fcak), cax2 = f2s(a.fcax);
        int it = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
            const int s = it % NSTv;
            const uint32_t ph = (uint32_t)(it / NSTv) & 1u;
            if (!mbar_wait(&full[s], ph, wait_lim)) {
                s_err = 1;
                break;
            }
            const TileInfo ti = load_info(&info[s]);
            const float* st = smem + (size_t)s * L::FLOATS;
            const int nx = ti.nx, ny = ti.ny;
            const int i0 = ti.x0 + c0;
            const int jt = ti.y0 + r0;
            if (i0 < nx && jt < ny) {
                if (ti.fs != 0 && jt < 9) {
#pragma unroll 1
                    for (int r = 0; r < NR; ++r) {
                        tma_point_scalar_t<R, BYv, HASU, HASA>(st, ti, a, c0, r0 + r, has_u, has_a);
                        tma_point_scalar_t<R, BYv, HASU, HASA>(st, ti, a, c0 + 1, r0 + r, has_u, has_a);
                    }
                } else {
                    const float* zvp = st + L::ZV_OFF;
                    const float* c2p = st + L::C2_OFF;
                    const float* wxp = st + L::WX_OFF;
                    const float* wyp = st + L::WY_OFF;
                    const float* yup = st + L::YU_OFF;
                    const float* spu = st + L::PU_OFF;
                    const float* spa = st + L::PA_OFF;
                    const bool fs = ti.fs != 0;
                    const bool in1 = i0 + 1 < nx;
                    const float* btab = ti.btab;
                    const int nbt = ti.nbtab;
                    // Where nothing damps the taps of this thread's points, z_x = z_y = 0 and the
                    // damping terms vanish (same results to the bit).
                    const bool damped = ti.xdamp || jt + NR + R >= ny - ti.pml || (!fs && jt - R <= ti.pml);
                    float2 bxn = f2s(0.f);
                    // bx at the half columns i0 + d + 1/2, d = -4 .. 5 (the z_x taps)
                    float bxh[10];
                    unsigned xin = 0u;                           // half columns 0 .. nx - 2
                    if (damped) {
                        bxn = f2(btab_at(btab, nbt, 2 * min(i0 + 1, nx - i0)),
                                 btab_at(btab, nbt, 2 * min(i0 + 2, nx - i0 - 1)));
#pragma unroll
                        for (int d = -4; d <= 5; ++d) {
                            const int p = i0 + d;
                            bxh[d + 4] = btab_at(btab, nbt, min(2 * p + 3, 2 * (nx - p) - 1));
                            if (p >= 0 && p < nx - 1) xin |= 1u << (d + 4);
                        }
                    }
                    // z_v = c^2 y_v and z_y = (bx - by^h) y_wy down this column pair
                    float2 zq[NR + 2 * R], zyq[NR + 2 * R - 1];
#pragma unroll
                    for (int q = 0; q < NR + 2 * R; ++q)
                        zq[q] = mul2(lds2(zvp + (r0 + q) * L::SW + cs), lds2(c2p + (r0 + q) * L::SW + cs));
                    if (damped) {
#pragma unroll
                        for (int q = 0; q < NR + 2 * R - 1; ++q) {
                            const int h = ti.y0 + r0 + q - R;
                            const float bh =
                                btab_at(btab, nbt, fs ? 2 * (ny - h) - 1 : min(2 * h + 3, 2 * (ny - h) - 1));
                            zyq[q] = (h >= 0 && h < ny - 1)
                                         ? mul2(sub2(bxn, f2s(bh)), lds2(wyp + (r0 + q) * BX + c0))
                                         : f2s(0.f);
                        }
                    }
                    const bool wx0in = i0 < nx - 1, wx1in = i0 + 1 < nx - 1;
                    const float2 idx1 = f2s(ti.idx1), idx2 = f2s(ti.idx2);
                    const float2 chx2 = f2s(a.fch * ti.xs);
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        const int lr = r0 + r, j = jt + r;
                        if (j >= ny) break;
                        // x taps of z_v (pairs at column offsets -4 .. 5)
                        const float* zr = zvp + (lr + R) * L::SW + cs;
                        const float* cr = c2p + (lr + R) * L::SW + cs;
                        const float2 zp[5] = {mul2(lds2(zr - 4), lds2(cr - 4)), mul2(lds2(zr - 2), lds2(cr - 2)),
                                              zq[r + R], mul2(lds2(zr + 2), lds2(cr + 2)),
                                              mul2(lds2(zr + 4), lds2(cr + 4))};
                        const float* wr = wxp + lr * L::SW + cs;
                        auto zo = [&](int d) { return ((d + 4) & 1) ? zp[(d + 4) >> 1].y : zp[(d + 4) >> 1].x; };
                        const float2 zc = zq[r + R];
                        float2 lap = mul2(f2s(2.f * cent<R>(0)), zc);
                        float2 dxt = f2s(0.f), dyt = f2s(0.f);
#pragma unroll
                        for (int k = 0; k < R; ++k) {
                            const int kk = k + 1;
                            const float2 sx = (kk & 1) ? f2(zo(kk) + zo(-kk), zo(kk + 1) + zo(1 - kk))
                                                       : add2(zp[(kk + 4) >> 1], zp[(4 - kk) >> 1]);
                            const float2 sy = add2(zq[r + R + kk], zq[r + R - kk]);
                            lap = fma2(f2s(cent<R>(kk)), add2(sx, sy), lap);
                            dxt = fma2(f2s(stag<R>(k)), f2(zo(-k) - zo(1 + k), zo(1 - k) - zo(2 + k)), dxt);
                            dyt = fma2(f2s(stag<R>(k)), sub2(zq[r + R + 1 + k], zq[r + R - k]), dyt);
                        }
                        const int pt = lr * BX + c0;
                        const float2 yv = lds2(zvp + (lr + R) * L::SW + cs);
                        const float2 yu = lds2(yup + pt);
                        if (ti.T) {
                            // grad += gscale y_v (L u + D w), the factor from the step's tape
                            const long long o = (long long)j * ti.pitch + i0;
                            const float2 gy = mul2(f2s((float)a.gscale), yv);
                            if (in1) {
                                const float2 g = *reinterpret_cast<const float2*>(ti.T + o);
                                float2* G = reinterpret_cast<float2*>(ti.G + o);
                                *G = add2(*G, mul2(gy, g));
                            } else {
                                ti.G[o] += gy.x * ti.T[o];
                            }
                        }
                        const bool wyin = j < ny - 1;
                        float2 ywx = lds2(wr);
                        if (!wx0in) ywx.x = 0.f;
                        if (!wx1in) ywx.y = 0.f;
                        const float2 ywy = wyin ? lds2(wyp + (lr + R) * BX + c0) : f2s(0.f);
                        // (H^T y)_u, _v, _wx, _wy
                        float2 hu, hv = yu, hwx, hwy = f2s(0.f);
                        if (damped) {
                            const float byn = btab_at(btab, nbt, 2 * (fs ? ny - j : min(j + 1, ny - j)));
                            const float byh =
                                btab_at(btab, nbt, fs ? 2 * (ny - j) - 1 : min(2 * j + 3, 2 * (ny - j) - 1));
                            // z_x at half column offset d: (by - bx^h) y_wx (zero off the w_x grid)
                            const float2 wp[5] = {lds2(wr - 4), lds2(wr - 2), lds2(wr), lds2(wr + 2), lds2(wr + 4)};
                            auto xo = [&](int d) {
                                const float wv = ((d + 4) & 1) ? wp[(d + 4) >> 1].y : wp[(d + 4) >> 1].x;
                                return ((xin >> (d + 4)) & 1u) ? (byn - bxh[d + 4]) * wv : 0.f;
                            };
                            float2 gxt = f2s(0.f), gyt = f2s(0.f);
#pragma unroll
                            for (int k = 0; k < R; ++k) {
                                gxt = fma2(f2s(stag<R>(k)), f2(xo(-1 - k) - xo(k), xo(-k) - xo(1 + k)), gxt);
                                gyt = fma2(f2s(stag<R>(k)), sub2(zyq[r + R + k], zyq[r + R - 1 - k]), gyt);
                            }
                            hu = fma2(mul2(bxn, f2s(-byn)), yv, fma2(lap, idx2, mul2(add2(gxt, gyt), idx1)));
                            hv = fma2(sub2(f2s(-byn), bxn), yv, yu);
                            hwx = fma2(dxt, idx1, mul2(f2(-bxh[4], -bxh[5]), ywx));
                            if (wyin) hwy = fma2(dyt, idx1, mul2(f2s(-byh), ywy));
                        } else {
                            hu = mul2(lap, idx2);
                            hwx = mul2(dxt, idx1);
                            if (wyin) hwy = mul2(dyt, idx1);
                        }
                        if (!wx0in) hwx.x = 0.f;
                        if (!wx1in) hwx.y = 0.f;
                        const float2 xf[4] = {yu, yv, ywx, ywy};
                        const float2 hf[4] = {hu, hv, hwx, hwy};
                        const long long o = (long long)j * ti.pitch + i0;
#pragma unroll
                        for (int f = 0; f < 4; ++f) {
                            const float2 uval = has_u ? lds2(spu + f * BYv * BX + pt) : f2s(0.f);
                            const float2 aval = has_a ? lds2(spa + f * BYv * BX + pt) : f2s(0.f);
                            const float2 kf = fma2(cx2, xf[f], mul2(chx2, hf[f]));
                            float2 yf = fma2(cu2, uval, mul2(ck2, kf));
                            float2 af = fma2(cax2, xf[f],
                                             fma2(cay2, yf, fma2(cak2, kf, fma2(cau2, uval, mul2(ca2, aval)))));
                            if (f == 2) {
                                if (!wx0in) yf.x = af.x = 0.f;
                                if (!wx1in) yf.y = af.y = 0.f;
                            }
                            if (f == 3 && !wyin) yf = af = f2s(0.f);
                            if (ti.Y) st2(ti.Y + f * ti.fstr + o, yf, in1);
                            if (ti.A) st2(ti.A + f * ti.fstr + o, af, in1);
                        }
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[s]);
        }
    }
    __syncthreads();
    tma_finish<NSTv>(s_err, issued, full, err);
}

// ---------------------------------------------------------------- host side
static PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

static int get_encoder() {
    if (g_encode) return 0;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
        return -1;
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    return 0;
}

// 4D map over (x, y, field, vector) of one buffer, box (bx, by, bf, 1).
static int encode4(CUtensorMap* out, void* base, int nx, int ny, int nvec, long long pitch,
                   long long fstride, long long vstride, int bx, int by, int bf) {
    cuuint64_t dims[4] = {(cuuint64_t)nx, (cuuint64_t)ny, 4, (cuuint64_t)nvec};
    cuuint64_t strides[3] = {(cuuint64_t)pitch * 4, (cuuint64_t)fstride * 4, (cuuint64_t)vstride * 4};
    cuuint32_t box[4] = {(cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bf, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = g_encode(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : -1;
}

static int encode2(CUtensorMap* out, void* base, int nx, int ny, long long pitch, int bx, int by) {
    cuuint64_t dims[2] = {(cuuint64_t)nx, (cuuint64_t)ny};
    cuuint64_t strides[1] = {(cuuint64_t)pitch * 4};
    cuuint32_t box[2] = {(cuuint32_t)bx, (cuuint32_t)by};
    cuuint32_t es[2] = {1, 1};
    CUresult r = g_encode(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : -1;
}

int tma_map_set(int tile_height) {
    for (int k = 0; k < TMA_NUM_SETS; ++k)
        if (TMA_SET_HEIGHTS[k] == tile_height) return k;
    return -1;
}
constexpr int map_set_of(int by) {
    for (int k = 0; k < TMA_NUM_SETS; ++k)
        if (TMA_SET_HEIGHTS[k] == by) return k;
    return -1;
}
static_assert(map_set_of(16) == 0 && map_set_of(18) == 3 && map_set_of(24) >= 0 && map_set_of(28) >= 0 &&
                  map_set_of(30) >= 0 && map_set_of(36) >= 0,
              "every tile height in use has a map set");

// Build NMAP maps per problem and tile height (one map set per entry of TMA_SET_HEIGHTS)
// into a device array (FP32 only); sets P.tmaps to the problem's first map.
int build_tensor_maps(std::vector<ProblemDev>& probs, int R, const std::vector<int>& work_vecs,
                      void** d_maps_inout) {
    if (get_encoder() != 0) return -1;
    const int n = (int)probs.size();
    constexpr int NSET = TMA_NUM_SETS;
    const int* heights = TMA_SET_HEIGHTS;
    std::vector<CUtensorMap> maps((size_t)n * NSET * NMAP);
    const int SW = BX + 2 * TX;
    for (int p = 0; p < n; ++p) {
        ProblemDev& P = probs[p];
        for (int set = 0; set < NSET; ++set) {
            const int by = heights[set], SH = by + 2 * R;
            CUtensorMap* m = maps.data() + ((size_t)p * NSET + set) * NMAP;
            const int bxs[5] = {SW, SW, BX, BX, BX};
            const int bys[5] = {SH, by, SH, by, by};
            const int bfs[5] = {1, 1, 1, 1, 4};
            for (int k = 0; k < 5; ++k) {
                if (encode4(m + k, P.state, P.nx, P.ny, 1, P.pitch, P.field_stride, P.vec_stride,
                            bxs[k], bys[k], bfs[k]) != 0)
                    return -1;
                void* wb = P.work ? P.work : P.state;
                const int nv = P.work ? work_vecs[p] : 1;
                if (encode4(m + 5 + k, wb, P.nx, P.ny, nv > 0 ? nv : 1, P.pitch, P.field_stride,
                            P.vec_stride, bxs[k], bys[k], bfs[k]) != 0)
                    return -1;
            }
            if (encode2(m + 10, const_cast<void*>(P.c2), P.nx, P.ny, P.pitch, BX, by) != 0) return -1;
            // c^2 with the 2D halo of u (the transposed pass stages c^2 y_v)
            if (encode2(m + 11, const_cast<void*>(P.c2), P.nx, P.ny, P.pitch, SW, SH) != 0) return -1;
        }
    }
    cudaFree(*d_maps_inout);
    *d_maps_inout = nullptr;
    if (cudaMalloc(d_maps_inout, sizeof(CUtensorMap) * maps.size()) != cudaSuccess) return -1;
    if (cudaMemcpy(*d_maps_inout, maps.data(), sizeof(CUtensorMap) * maps.size(),
                   cudaMemcpyHostToDevice) != cudaSuccess)
        return -1;
    for (int p = 0; p < n; ++p)
        probs[p].tmaps = static_cast<char*>(*d_maps_inout) + (size_t)p * NSET * NMAP * sizeof(CUtensorMap);
    return 0;
}

// Kernel variants the autotuner chooses from: (tile height, consumer warps, stages).  One row a
// thread where the warps equal the rows, else two (variant 12 four).  Variant 4 has no U buffer
// (4 stages of 64 x 16): passes with a U operand run variant 0 instead.  11 to 14 are composite:
// passes that read an A operand run variant 7, the others (Horner HORK passes, Krylov products,
// leap-frog-free RK stages without an accumulator) drop the A buffer and take taller tiles (14:
// 512 threads at 128 registers, the whole register file).  The shape reported for a composite is
// its no-A shape.  Variant 10, two stages with the A buffer, is the better A shape where a pass is
// a few tiles per SM (16 shots of 401 x 201: 20 us against 22 of variant 7), but without an A
// operand it lost to 14 there (21 against 18): those passes run 14's shape.
struct TmaVariant {
    int by, nw, nst;
};
constexpr TmaVariant kVariants[TMA_NUM_VARIANTS] = {
    {16, 16, 3}, {16, 8, 3}, {8, 8, 5},  {8, 4, 5},  {16, 16, 4}, {20, 10, 3}, {18, 18, 3},
    {18, 9, 3},  {16, 8, 3}, {18, 18, 3}, {24, 12, 2}, {24, 12, 3}, {36, 9, 2}, {28, 14, 3}, {30, 15, 3}};

static bool composite(int v) { return v >= 11 && v <= 14; }

// A pass with an A operand and no U (the low-storage HORK stages) needs as many stage buffers as
// one with U and no A: the composite variants and 10 run it on 14's tall tiles.  HORK 20, 16 shots of
// 803 x 397: 1240 us a step (24 rows with both buffers and two stages: 1272; variant 7's shape: 1302).
static bool a_only_on_tall(int v, bool reads_u, bool reads_a) {
    return (composite(v) || v == 10) && reads_a && !reads_u;
}

constexpr int A_ONLY_TALL = TMA_NUM_VARIANTS;   // (64 x 30, 15 warps, 3 stages, no U buffer)
int tma_variant_shape(int v) { return v == 1 ? 8 : v == 6 ? 9 : v; }
int tma_pass_shape(int v, bool reads_u, bool reads_a) {
    if (a_only_on_tall(v, reads_u, reads_a)) return A_ONLY_TALL;
    if (composite(v) && reads_a) return 7;
    if (v == 10 && !reads_a) return 14;
    if (v == 4 && reads_u) return 0;                // no U buffer
    return tma_variant_shape(v);
}
int tma_variant_tile_height_for(int v, bool reads_u, bool reads_a) {
    const int shape = tma_pass_shape(v, reads_u, reads_a);
    return shape == A_ONLY_TALL ? 30 : kVariants[shape].by;
}

int tma_variant_tile_height(int v) { return kVariants[v].by; }
// The pass that writes a gradient tape reads no A operand, so it runs on 14's tall tiles where one of
// the small shapes below 7 is selected (same bits on every shape).  FWI gradient, Horner HORK 20, 16
// shots of 401 x 201, on 14's shape and on the selected one: 12.8 and 13.7 ms (variant 0), 14.1 and
// 16.2 (2), 14.0 and 16.0 (3), 12.5 and 13.2 (5); on 2 shots of 301 x 151, whose tiles do not fill the
// chip either way, 4.46 and 4.29 ms (0), 4.53 and 4.41 (2).
int tma_tape_variant(int v) { return v >= 7 ? v : 14; }
void tma_variant_describe(int v, int* by, int* nw, int* nst) {
    *by = kVariants[v].by;
    *nw = kVariants[v].nw;
    *nst = kVariants[v].nst;
}

static int g_num_sms = 0;

// Dynamic shared memory of a launch: only the stages that a block's tiles touch.  On small grids that
// leaves room for the next pass's block beside this one (pdl.cuh).
static size_t smem_in_use(size_t all, int stages, int ntiles, int grid) {
    const int per = (ntiles + grid - 1) / grid;
    return per >= stages ? all : (all - 1024) / stages * per + 1024;
}

template <int R, int BYv, int NW, int NSTv, int EPI, bool HASA = true, bool HASU = true>
static int launch_x2(const ProblemDev* probs, const int* tbase, int nprob, int ntiles, const StageArgs& a,
                     int* err, cudaStream_t s) {
    static_assert(map_set_of(BYv) >= 0, "tile height without a map set");
    if (!HASA && a.a >= 0) return -1;    // a pass with an A operand needs the A buffer
    if (!HASU && a.u >= 0) return -1;    // and one with a U operand the U buffer
    const size_t smem = (size_t)NSTv * StageLayout<R, BYv, HASU, HASA>::BYTES + 1024;
    static unsigned long long configured = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
    if (!(configured >> dev & 1ull)) {
        if (cudaFuncSetAttribute(stage_tma_x2_kernel<R, BYv, NW, NSTv, EPI, HASU, HASA>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return -1;
        configured |= 1ull << dev;
    }
    const int grid = ntiles < g_num_sms ? ntiles : g_num_sms;
    const size_t used = smem_in_use(smem, NSTv, ntiles, grid);
    return launch_pdl(stage_tma_x2_kernel<R, BYv, NW, NSTv, EPI, HASU, HASA>, grid, NW * 32 + 32, used, s, probs, tbase,
                      nprob, ntiles, map_set_of(BYv), a, err);
}

// One leap-frog step (EPI 2) on the column-pair consumers (64 x 30 tiles, 15 warps, 3
// stages, no U buffer); tbase and ntiles are those of the 30-row map set.
int launch_leapfrog_tma(int R, const ProblemDev* probs, const int* tbase, int nprob, int ntiles, int cur,
                        int prev, int variant, double dt, int* err, cudaStream_t s) {
    if (ntiles <= 0) return nprob > 0 ? -1 : 0;
    if (!g_num_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_num_sms <= 0) g_num_sms = 1;
    }
    StageArgs a{};
    a.x = cur;
    a.u = -1;
    a.a = prev;
    a.y_out = prev;
    a.acc_out = cur;
    a.d = -1;
    a.src_slot = 0;
    a.x_scale_slot = -1;
    a.m = variant;
    a.dt = dt;
    if (R == 4) return launch_x2<4, 30, 15, 3, 2, true, false>(probs, tbase, nprob, ntiles, a, err, s);
    if (R == 2) return launch_x2<2, 30, 15, 3, 2, true, false>(probs, tbase, nprob, ntiles, a, err, s);
    return -1;
}

// The FWI gradient pass (EPI 3): grad += gscale q_v (L u + D w) of vector a.x, q = a.gq (its
// four fields ride in the A box); column-pair consumers on the leap-frog step's tiles
// (64 x 30, 15 warps, 3 stages; the 30-row map set).
int launch_grad_tma(int R, const ProblemDev* probs, const int* tbase, int nprob, int ntiles,
                    const StageArgs& a_in, int* err, cudaStream_t s) {
    if (ntiles <= 0) return nprob > 0 ? -1 : 0;
    if (!g_num_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_num_sms <= 0) g_num_sms = 1;
    }
    StageArgs a = a_in;
    a.u = -1;
    a.a = a.gq;
    a.y_out = -1;
    a.acc_out = -1;
    if (R == 4) return launch_x2<4, 30, 15, 3, 3, true, false>(probs, tbase, nprob, ntiles, a, err, s);
    if (R == 2) return launch_x2<2, 30, 15, 3, 3, true, false>(probs, tbase, nprob, ntiles, a, err, s);
    return -1;
}

template <int R, int BYv, int NW, int NSTv, bool HASU, bool HASA>
static int launch_t(const ProblemDev* probs, const int* tbase, int nprob, int ntiles, const StageArgs& a, int* err,
                    cudaStream_t s) {
    static_assert(map_set_of(BYv) >= 0, "tile height without a map set");
    const size_t smem = (size_t)NSTv * TLayout<R, BYv, HASU, HASA>::BYTES + 1024;
    static unsigned long long configured = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
    if (!(configured >> dev & 1ull)) {
        if (cudaFuncSetAttribute(stage_tma_t_kernel<R, BYv, NW, NSTv, HASU, HASA>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return -1;
        configured |= 1ull << dev;
    }
    const int grid = ntiles < g_num_sms ? ntiles : g_num_sms;
    const size_t used = smem_in_use(smem, NSTv, ntiles, grid);
    return launch_pdl(stage_tma_t_kernel<R, BYv, NW, NSTv, HASU, HASA>, grid, NW * 32 + 32, used, s, probs, tbase, nprob,
                      ntiles, map_set_of(BYv), a, err);
}

// The transposed pass H^T (FP32; with a tape set, the gradient too) on the column-pair consumers, two
// rows a thread.  The tile is as tall as three stages fit shared memory, since the consumer warps hide
// the latency: 64 x 18 with 9 warps for a pass with a U and an A operand, 64 x 24 with 12 for one of
// them, 64 x 30 with 15 for the plain product; tbase and ntiles are those of that height's map set.
int tma_transpose_height(bool reads_u, bool reads_a) { return reads_u && reads_a ? 18 : reads_u || reads_a ? 24 : 30; }
int launch_transpose_tma(int R, const ProblemDev* probs, const int* tbase, int nprob, int ntiles,
                         const StageArgs& a_in, int* err, cudaStream_t s) {
    if (ntiles <= 0) return nprob > 0 ? -1 : 0;
    if (!g_num_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_num_sms <= 0) g_num_sms = 1;
    }
    StageArgs a = a_in;
    a.fcx = (float)a.cx;
    a.fch = (float)a.ch;
    a.fcu = (float)a.cu;
    a.fck = (float)a.ck;
    a.fca = (float)a.ca;
    a.fcau = (float)a.cau;
    a.fcak = (float)a.cak;
    a.fcay = (float)a.cay;
    a.fcax = (float)a.cax;
    const bool hu = a.u >= 0, ha = a.a >= 0;
    if (R == 4) {
        if (hu && ha) return launch_t<4, 18, 9, 3, true, true>(probs, tbase, nprob, ntiles, a, err, s);
        if (hu) return launch_t<4, 24, 12, 3, true, false>(probs, tbase, nprob, ntiles, a, err, s);
        if (ha) return launch_t<4, 24, 12, 3, false, true>(probs, tbase, nprob, ntiles, a, err, s);
        return launch_t<4, 30, 15, 3, false, false>(probs, tbase, nprob, ntiles, a, err, s);
    }
    if (R == 2) {
        if (hu && ha) return launch_t<2, 18, 9, 3, true, true>(probs, tbase, nprob, ntiles, a, err, s);
        if (hu) return launch_t<2, 24, 12, 3, true, false>(probs, tbase, nprob, ntiles, a, err, s);
        if (ha) return launch_t<2, 24, 12, 3, false, true>(probs, tbase, nprob, ntiles, a, err, s);
        return launch_t<2, 30, 15, 3, false, false>(probs, tbase, nprob, ntiles, a, err, s);
    }
    return -1;
}

int launch_stage_tma(int variant, int R, const ProblemDev* probs, const int* tbase, int nprob,
                     int ntiles, const StageArgs& a_in, int* err, cudaStream_t s) {
    StageArgs a = a_in;
    a.fcx = (float)a.cx;
    a.fch = (float)a.ch;
    a.fcu = (float)a.cu;
    a.fck = (float)a.ck;
    a.fca = (float)a.ca;
    a.fcau = (float)a.cau;
    a.fcak = (float)a.cak;
    a.fcay = (float)a.cay;
    a.fcax = (float)a.cax;
    if (ntiles <= 0) return nprob > 0 ? -1 : 0;   // problems but no tiles: inconsistent lists
    if (a.tape_vec > 0 && (tma_tape_variant(variant) != variant || a.a >= 0)) return -1;
    if (!g_num_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_num_sms <= 0) g_num_sms = 1;
    }
    // the steady-state Faber / HORK form: Y = cu U + cx X + ch H, ACC = ca A + cay Y
    const bool epi = a.ck == 1.0 && a.cau == 0.0 && a.cak == 0.0 && a.cax == 0.0;
    variant = tma_pass_shape(variant, a.u >= 0, a.a >= 0);
#define EWV_TMA_CASE2(V, RR, BYV, NWV, NSTV, HASA, HASU)                                                   \
    if (variant == V && R == RR)                                                                         \
        return epi ? launch_x2<RR, BYV, NWV, NSTV, 1, HASA, HASU>(probs, tbase, nprob, ntiles, a, err, s) \
                   : launch_x2<RR, BYV, NWV, NSTV, 0, HASA, HASU>(probs, tbase, nprob, ntiles, a, err, s);
#define EWV_TMA_CASE(V, BYV, NWV, NSTV, HASA, HASU)  \
    EWV_TMA_CASE2(V, 4, BYV, NWV, NSTV, HASA, HASU) \
    EWV_TMA_CASE2(V, 2, BYV, NWV, NSTV, HASA, HASU)
    EWV_TMA_CASE(A_ONLY_TALL, 30, 15, 3, true, false)
    EWV_TMA_CASE(0, 16, 16, 3, true, true)
    EWV_TMA_CASE(2, 8, 8, 5, true, true)
    EWV_TMA_CASE(3, 8, 4, 5, true, true)
    EWV_TMA_CASE(4, 16, 16, 4, true, false)
    EWV_TMA_CASE(5, 20, 10, 3, true, true)
    EWV_TMA_CASE(7, 18, 9, 3, true, true)
    EWV_TMA_CASE(8, 16, 8, 3, true, true)
    EWV_TMA_CASE(9, 18, 18, 3, true, true)
    EWV_TMA_CASE(10, 24, 12, 2, true, true)
    EWV_TMA_CASE(11, 24, 12, 3, false, true)
    EWV_TMA_CASE(12, 36, 9, 2, false, true)
    EWV_TMA_CASE(13, 28, 14, 3, false, true)
    EWV_TMA_CASE(14, 30, 15, 3, false, true)
#undef EWV_TMA_CASE
#undef EWV_TMA_CASE2
    return -1;
}

}  // namespace ewv
