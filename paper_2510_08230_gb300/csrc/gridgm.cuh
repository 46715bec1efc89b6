// gridgm.cuh - GMRES(m) (none or Jacobi) as one persistent cooperative kernel
// over the whole GPU, for matrices whose solver layout is ELL.
//
// The method is the multi-kernel engine's: right preconditioning, classical
// Gram-Schmidt applied twice, Givens rotations, the estimate checked after
// every Arnoldi step, every cycle started from the true residual.  There a
// step is seven kernels; on the 128^3 diffusion matrix (16 columns) the three
// passes over the basis took 353 us for 216 us of FP64 work: 28 % and 14 %
// more FP64 instructions than products (a five-level shuffle tree per column
// and 2048-row chunk), 10 to 20 us a kernel of ticket, last block and serial
// Givens arithmetic on global memory.
//
// Here a block keeps w (its rows) in shared memory and streams its rows of
// the basis three times a step: h1 = V^T w; w -= V h1, h2 = V^T w;
// w -= V h2, ||w||.  A thread takes four columns of four of its rows at a time
// (16 loads in flight); a warp's 4 x 32 partial sums of four columns collapse
// with six adds (a shuffle level serves all of them).  The k + 1
// sums are handed over together, the Givens step runs in every block on
// shared memory, and only z = M^-1 v_k is published.
//
// Per step of Jacobi-GMRES(30), multi-kernel / this kernel (GB300, us): FP64
// 10,000-row 2D stencil 99 / 35, 117,000-row 3D stencil 105 / 50, 10^6 rows
// 252 / 182, 128^3 diffusion 407 / 328 (the FP64 pipe's floor 247); FP32 53 /
// 34, 62 / 36, 111 / 74, 185 / 133.  At 128^3 a step's 680,000 cycles are
// 260,000 in the two passes of products, 247,000 in the two updates and
// 85,000 in the SpMV; on small matrices they are hand-offs and the serial
// Givens step.  Tried: eight columns a pass with one row (903,000 cycles: a
// 5-level shuffle tree per column and row block), the passes inlined into the
// step's loop (spills at 64 registers: 908,000).
// Six solves of 70K to 430K rows at once, 240 steps each, ms: FP64 65 / 86 to
// 106 (alone, in turn: 167 / 94), FP32 28 / 51 (93 / 58).  Two grids are
// resident together and gain little on each other, since a step's folds, Givens
// arithmetic and hand-offs keep every SM's FP64 pipe, whatever the type; the
// multi-kernel engine does the serial part on one SM.  Fewer, larger blocks
// (3,072 rows at least) would give 32 at once in FP32, but 11.0 to 11.5 ms alone
// instead of 8.6 to 11.1.
#pragma once

#include "gridbase.cuh"

namespace gk {

template <typename V, typename T>
struct GridGmArgs {
    int32_t n, R, K, m;
    int64_t stride;
    const int32_t* col;
    const V* val;
    const T* b;
    T* x;           // the iterate (padded to whole blocks)
    const T* x0;
    const T* dinv;  // null: no preconditioner
    T* p;           // gathered vector, padded to whole blocks
    T* basis;       // m + 1 columns of ldv entries
    int64_t ldv;
    unsigned long long *slots, *arrived;
    int32_t* err;
    GridOut* out;
    double tol;
    int32_t max_iters;
    double stag;    // > 0: stop when a cycle's residual exceeds stag x the previous
    uint64_t wait_ns;
    unsigned between;  // see GridTeam
};

// Shared memory: the scalar sums, each warp's column sums, h1, h2, the triangular
// factor, cs, sn, g, the coefficients of the update under way (in T), w, and
// the matrix rows.
template <int NT>
__host__ __device__ inline size_t grid_gm_fixed(int m) {
    const size_t nc = (size_t)m + 1;
    return GRID_RED<NT> + 8 * (NT / 32 * nc + 2 * nc + (size_t)m * m + 4 * nc);
}
template <int NT, typename V, typename T>
size_t grid_gm_smem(bool staged, int m, int64_t R, int64_t K) {
    return ((grid_gm_fixed<NT>(m) + 15) & ~(size_t)15) + (size_t)R * sizeof(T) +
           (staged ? (size_t)(R * K) * (sizeof(V) + 4) : 0);
}

// Sums 4 values over the warp: lane l holds the total of value l >> 3.
__device__ __forceinline__ double warp_sum4(const double (&a)[4]) {
    const int lane = threadIdx.x & 31;
    double b[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const bool hi = (lane & 16) != 0;
        b[i] = (hi ? a[i + 2] : a[i]) + __shfl_xor_sync(0xffffffffu, hi ? a[i] : a[i + 2], 16);
    }
    const bool hi = (lane & 8) != 0;
    double t = (hi ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, hi ? b[0] : b[1], 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// Givens step on column k of a cycle: applies the rotations so far to its
// entries h1 + h2 and hk1 (column k of the factor goes to tri), appends the
// next one and updates g.  Returns 0, END_NAN or END_BREAKDOWN; *est: the
// residual estimate.  Not inlined: its registers are not the hot loops'.
static __device__ __noinline__ int givens_step(int k, double hk1, const double* h1, const double* h2,
                                               double* tri, double* cs, double* sn, double* g,
                                               double* est) {
    double cur = h1[0] + h2[0];
    for (int j = 0; j < k; ++j) {
        const double nxt = h1[j + 1] + h2[j + 1];
        const double c = cs[j], s = sn[j];
        tri[j] = c * cur + s * nxt;
        cur = -s * cur + c * nxt;
    }
    const double d = hypot(cur, hk1);
    if (!isfinite(d)) return END_NAN;
    if (d == 0.0) return END_BREAKDOWN;
    cs[k] = cur / d;
    sn[k] = hk1 / d;
    tri[k] = d;
    g[k + 1] = -sn[k] * g[k];
    g[k] = cs[k] * g[k];
    *est = fabs(g[k + 1]);
    return isfinite(*est) ? 0 : END_NAN;
}

// The passes over the basis.  Not inlined: each gets the registers for 16
// loads in flight, and what the solve keeps live is saved once per call.
// v: the block's first row of column 0.
template <typename T>
struct GmBasis {
    T* v;
    int64_t ldv;
    int32_t nloc;
};

// acc[u] += the products of NC columns (pointers q at row li) with NR of the
// thread's rows of w
template <int NT, int NR, int NC, typename T>
__device__ __forceinline__ void gm_dots_block(const T* const (&q)[NC], const T* w, T (&acc)[NC]) {
    T v[NR][NC];
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int u = 0; u < NC; ++u) v[r][u] = __ldcg(q[u] + r * NT);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const T wv = w[r * NT];
#pragma unroll
        for (int u = 0; u < NC; ++u) acc[u] = fmadd(v[r][u], wv, acc[u]);
    }
}

// the warp's parts of NC columns from c0 on
template <int NT, int NC, typename T>
__device__ __forceinline__ void gm_dots_columns(const GmBasis<T>& B, const T* ws, int c0, double* out) {
    T acc[NC];
    const T* q[NC];
#pragma unroll
    for (int u = 0; u < NC; ++u) {
        acc[u] = T(0);
        q[u] = B.v + (c0 + u) * B.ldv + threadIdx.x;
    }
    int32_t li = threadIdx.x;
    auto step = [&](auto nr) {
        constexpr int NR = decltype(nr)::value;
        gm_dots_block<NT, NR, NC, T>(q, ws + li, acc);
        li += NR * NT;
#pragma unroll
        for (int u = 0; u < NC; ++u) q[u] += NR * NT;
    };
    if constexpr (NC <= 4) {
        while (li + 3 * NT < B.nloc) step(std::integral_constant<int, 4>{});
        if (li + NT < B.nloc) step(std::integral_constant<int, 2>{});
    }
    if (li < B.nloc) step(std::integral_constant<int, 1>{});
    const int lane = threadIdx.x & 31;
    if constexpr (NC % 4 == 0) {
#pragma unroll
        for (int g = 0; g < NC; g += 4) {
            const double d[4] = {(double)acc[g], (double)acc[g + 1], (double)acc[g + 2], (double)acc[g + 3]};
            const double t = warp_sum4(d);
            if ((lane & 7) == 0) out[c0 + g + (lane >> 3)] = t;
        }
    } else {
#pragma unroll
        for (int u = 0; u < NC; ++u) {
            const double t = warp_sum((double)acc[u]);
            if (lane == 0) out[c0 + u] = t;
        }
    }
}

// out[c] = this warp's part of <v_c, w>, c < ncol
template <int NT, typename T>
__device__ __noinline__ void gm_column_dots(GmBasis<T> B, const T* ws, int ncol, double* out) {
    int c0 = 0;
    if (B.nloc <= NT)  // one row a thread: the loads in flight are columns
        for (; c0 + 8 <= ncol; c0 += 8) gm_dots_columns<NT, 8, T>(B, ws, c0, out);
    for (; c0 + 4 <= ncol; c0 += 4) gm_dots_columns<NT, 4, T>(B, ws, c0, out);
    if (ncol - c0 >= 2) {
        gm_dots_columns<NT, 2, T>(B, ws, c0, out);
        c0 += 2;
    }
    if (c0 < ncol) gm_dots_columns<NT, 1, T>(B, ws, c0, out);
}

// NR rows of w from li on: w += V coef, in column order; adds to the sum of squares
template <int NT, int NR, typename T>
__device__ __forceinline__ T gm_update_rows(const GmBasis<T>& B, T* w, const T* coef, int ncol,
                                            int32_t li, T sq) {
    T wv[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) wv[r] = w[li + r * NT];
    constexpr int NC = NR == 1 ? 8 : 4;
    const T* q = B.v + li;
    int c = 0;
    for (; c + NC <= ncol; c += NC) {
        T v[NC][NR];
#pragma unroll
        for (int u = 0; u < NC; ++u) {
#pragma unroll
            for (int r = 0; r < NR; ++r) v[u][r] = __ldcg(q + r * NT);
            q += B.ldv;
        }
#pragma unroll
        for (int u = 0; u < NC; ++u) {
            const T h = coef[c + u];
#pragma unroll
            for (int r = 0; r < NR; ++r) wv[r] = fmadd(h, v[u][r], wv[r]);
        }
    }
    for (; c < ncol; ++c, q += B.ldv) {
        const T h = coef[c];
        T v[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) v[r] = __ldcg(q + r * NT);
#pragma unroll
        for (int r = 0; r < NR; ++r) wv[r] = fmadd(h, v[r], wv[r]);
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        w[li + r * NT] = wv[r];
        sq = fmadd(wv[r], wv[r], sq);
    }
    return sq;
}

// w += V coef; the thread's sum of squares
template <int NT, typename T>
__device__ __noinline__ T gm_update(GmBasis<T> B, T* ws, const T* coef, int ncol) {
    T sq = T(0);
    int32_t li = threadIdx.x;
    for (; li + 3 * NT < B.nloc; li += 4 * NT) sq = gm_update_rows<NT, 4, T>(B, ws, coef, ncol, li, sq);
    if (li + NT < B.nloc) {
        sq = gm_update_rows<NT, 2, T>(B, ws, coef, ncol, li, sq);
        li += 2 * NT;
    }
    if (li < B.nloc) sq = gm_update_rows<NT, 1, T>(B, ws, coef, ncol, li, sq);
    return sq;
}

// w = (the block's rows of A) p
template <int NT, typename V, typename T, bool STAGED>
__device__ __noinline__ void gm_product(const GridRows<NT, V, T, STAGED>& rows, const T* p, T* ws) {
    rows.product(p, [&](int32_t li, T s) { ws[li] = s; });
}

template <int NT, typename V, typename T, bool STAGED, bool PREC>
__global__ void __launch_bounds__(NT, GRID_FULL / NT) k_grid_gmres(const GridGmArgs<V, T> A) {
    constexpr int NW = NT / 32;
    extern __shared__ __align__(128) unsigned char smem[];
    const int m = A.m, nc = m + 1;
    const int32_t R = A.R;
    double* s_part = reinterpret_cast<double*>(smem + GRID_RED<NT>);  // [NW][nc]
    double* s_h1 = s_part + NW * nc;
    double* s_h2 = s_h1 + nc;
    double* s_tri = s_h2 + nc;  // column k of the triangular factor at k m
    double* s_cs = s_tri + m * m;
    double* s_sn = s_cs + nc;
    double* s_g = s_sn + nc;
    T* s_coef = reinterpret_cast<T*>(s_g + nc);
    T* ws = reinterpret_cast<T*>(smem + ((grid_gm_fixed<NT>(m) + 15) & ~(size_t)15));
    V* s_val = reinterpret_cast<V*>(ws + R);
    __shared__ double part[8];
    __shared__ int s_code;
    __shared__ struct {
        double bn, thr, tn, prev, rec, inv;
    } S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t r0 = (int32_t)blockIdx.x * R;
    const int32_t nloc = min(R, A.n - r0);  // >= 1
    GridTeam<NT> team{A.slots, A.arrived, A.err, A.wait_ns, A.between, (int)gridDim.x, nc, nloc > NT / 2,
                  reinterpret_cast<double*>(smem), part, &s_code, 0u};
    const GridRows<NT, V, T, STAGED> rows{R, A.K, r0, nloc, A.stride, A.col, A.val, s_val,
                                          reinterpret_cast<int32_t*>(s_val + (size_t)(STAGED ? R * A.K : 0))};
    const GmBasis<T> basis{A.basis + r0, A.ldv, nloc};
    rows.stage();
    for (int32_t li = tid; li < nloc; li += NT) A.p[r0 + li] = A.x[r0 + li] = A.x0[r0 + li];

    // s_part[0][c] = sum over the warps' s_part[.][c], in two levels
    auto fold_parts = [&](int ncol) {
        __syncthreads();
        for (int level = 0; level < 2; ++level) {
            // 8 warps add PW each (into rows 0, PW, ...), then one adds those 8
            constexpr int PW = NW / 8;
            static_assert(PW <= 4, "the first level adds up to four");
            const int step = level == 0 ? 1 : PW, count = level == 0 ? PW : 8;
            const int lead = level == 0 ? PW * warp : 0;
            if (warp < (level == 0 ? 8 : 1))
                for (int c = lane; c < ncol; c += 32) {
                    double t[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        t[q] = q < count ? s_part[(lead + q * step) * nc + c] : 0.0;
                    s_part[lead * nc + c] = level == 0
                                                ? (t[0] + t[1]) + (t[2] + t[3])
                                                : ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
                }
            __syncthreads();
        }
    };
    // h[c] = <v_c, w> over the grid, s_coef[c] = -h[c], c < ncol; which: the
    // round's vector slots
    auto grid_dots = [&](int ncol, int which, double* h) -> bool {
        gm_column_dots<NT, T>(basis, ws, ncol, s_part + warp * nc);
        fold_parts(ncol);
        unsigned long long* sl = team.vslot(team.round, which);
        if (warp == 0)
            for (int c = lane; c < ncol; c += 32)
                post_slot(sl + (size_t)blockIdx.x * nc + c, s_part[c]);
        if (tid == 0) s_code = 0;
        __syncthreads();
        // warp w adds the sums of blocks w, w + NW, ...; lanes over columns
        for (int cb = 0; cb < ncol; cb += 32) {
            const int c = cb + lane;
            double x = 0.0;
#pragma unroll
            for (int b0 = 0; b0 < GRID_MAX_BLOCKS; b0 += GRID_POLLS * NW) {
                unsigned long long u[GRID_POLLS];
                const bool ok = team.wait([&] {
                    bool all = true;
#pragma unroll
                    for (int j = 0; j < GRID_POLLS; ++j) {
                        const int bk = b0 + warp + NW * j;
                        u[j] = bk < team.nb && c < ncol ? ld_slot(sl + (size_t)bk * nc + c) : 0ull;
                    }
#pragma unroll
                    for (int j = 0; j < GRID_POLLS; ++j) all &= u[j] != SLOT_EMPTY;
                    return all;
                });
                if (!ok && lane == 0) s_code = END_TIMEOUT;
                double y[GRID_POLLS];
#pragma unroll
                for (int j = 0; j < GRID_POLLS; ++j) y[j] = __longlong_as_double((long long)u[j]);
                x += ((y[0] + y[1]) + (y[2] + y[3])) + y[4];
            }
            if (c < ncol) s_part[warp * nc + c] = x;
        }
        fold_parts(ncol);
        for (int c = tid; c < ncol; c += NT) {
            h[c] = s_part[c];
            s_coef[c] = -(T)s_part[c];
        }
        __syncthreads();
        return s_code == 0;
    };
    // v_k = w * S.inv ; z = M^-1 v_k, published
    auto next_vector = [&](int k) -> bool {
        const T ih = (T)S.inv;
        rows.each([&](int32_t li) {
            const T v = ws[li] * ih;
            basis.v[k * A.ldv + li] = v;
            A.p[r0 + li] = PREC ? A.dinv[r0 + li] * v : v;
        });
        rows.prefetch_first();
        return team.publish();
    };
    int iters = 0, restarts = 0, k = 0;
    bool cycled = false;
    // w = b - A x for the x published in A.p, and what the cycle's start decides
    auto start_cycle = [&](bool first) -> int {
        T a[2] = {T(0), T(0)};
        rows.product(A.p, [&](int32_t li, T s) {
            const T bi = A.b[r0 + li];
            const T ri = bi - s;
            ws[li] = ri;
            a[0] = fmadd(bi, bi, a[0]);
            a[1] = fmadd(ri, ri, a[1]);
        });
        const double v[2] = {(double)a[0], (double)a[1]};
        const int end = team.sum<2>(0, v, [&](const double* t) -> int {
            if (first) {
                S.bn = sqrt(t[0]);
                S.thr = A.tol * S.bn;
                S.prev = S.rec = 0.0;
                if (!isfinite(S.bn)) return END_NAN;
                if (S.bn == 0.0) return END_ZERO;
            }
            const double b0 = sqrt(t[1]);
            S.tn = b0;
            if (!isfinite(b0)) return END_NAN;
            if (b0 <= S.thr) return END_OK;
            if (iters >= A.max_iters) return END_CAP;
            if (A.stag > 0.0 && S.prev > 0.0 && b0 > A.stag * S.prev) return END_CAP;
            S.prev = b0;
            s_g[0] = b0;
            S.inv = 1.0 / b0;
            return 0;
        });
        if (end == 0 && cycled) restarts += 1;
        k = 0;
        return end;
    };

    int end = team.publish() ? start_cycle(true) : END_TIMEOUT;
    if (end == 0 && !next_vector(0)) end = END_TIMEOUT;
    while (end == 0) {
        gm_product(rows, A.p, ws);
        const int ncol = k + 1;
        if (!grid_dots(ncol, 0, s_h1)) { end = END_TIMEOUT; break; }
        gm_update<NT, T>(basis, ws, s_coef, ncol);
        if (!grid_dots(ncol, 1, s_h2)) { end = END_TIMEOUT; break; }
        const double v[1] = {(double)gm_update<NT, T>(basis, ws, s_coef, ncol)};
        // Givens step on column k, the residual estimate, the cycle's end
        end = team.sum<1>(1, v, [&](const double* t) -> int {
            const double hk1 = sqrt(t[0]);
            double est = 0.0;
            const int bad = givens_step(k, hk1, s_h1, s_h2, s_tri + k * m, s_cs, s_sn, s_g, &est);
            if (bad) return bad;
            S.rec = est;
            if (hk1 == 0.0 || est <= S.thr || k + 1 == m || iters + 1 >= A.max_iters)
                return CYCLE;
            S.inv = 1.0 / hk1;
            return 0;
        });
        if (end != 0 && end != CYCLE) break;
        ++iters;
        k += 1;
        if (end == 0) {
            if (!next_vector(k)) end = END_TIMEOUT;
            continue;
        }
        // cycle end: y = R^-1 g (lane l of warp 0 holds g_l and g_{l+32}),
        // x += M^-1 (V y), and the next cycle from the true residual
        if (warp == 0) {
            double g0 = lane < k ? s_g[lane] : 0.0, g1 = lane + 32 < k ? s_g[lane + 32] : 0.0;
            for (int i = k - 1; i >= 0; --i) {
                const double gi = __shfl_sync(0xffffffffu, i < 32 ? g0 : g1, i & 31);
                const double yi = gi / s_tri[i * m + i];
                if (lane == 0) s_coef[i] = (T)yi;
                if (lane < i) g0 = fma(-s_tri[i * m + lane], yi, g0);
                if (lane + 32 < i) g1 = fma(-s_tri[i * m + lane + 32], yi, g1);
            }
        }
        __syncthreads();
        rows.each([&](int32_t li) { ws[li] = T(0); });
        gm_update<NT, T>(basis, ws, s_coef, k);
        rows.each([&](int32_t li) {
            const T xi = PREC ? fmadd(A.dinv[r0 + li], ws[li], A.x[r0 + li]) : A.x[r0 + li] + ws[li];
            A.x[r0 + li] = xi;
            A.p[r0 + li] = xi;
        });
        cycled = true;
        end = team.publish() ? start_cycle(false) : END_TIMEOUT;
        if (end == 0 && !next_vector(0)) end = END_TIMEOUT;
    }
    if (end == END_ZERO)
        for (int32_t li = tid; li < nloc; li += NT) A.x[r0 + li] = T(0);
    if (blockIdx.x == 0 && tid == 0) {
        GridOut o;
        o.status = end_status(end);
        o.iters = iters;
        o.restarts = restarts;
        o.pad = 0;
        o.rec = S.bn > 0.0 ? S.rec / S.bn : 0.0;
        o.tru = S.bn > 0.0 ? S.tn / S.bn : 0.0;
        *A.out = o;
    }
}

// ------------------------------------------------------------ host side

// One GMRES(m) solve on k_grid_gmres.  GK_ERR_UNSUPPORTED, with x untouched: a
// block's rows of w do not fit its shared memory, there is no room for the
// basis, the grid cannot be resident at once, or a wait ran out.
template <typename V, typename T>
gk_status solve_grid_gmres(gk_matrix M, const T* b, T* x, int pkind, double tol, int32_t max_iters,
                           int m, cudaStream_t s, SolveOut* out, bool inner) {
    const int32_t n = M->n;
    SolverCache* C = nullptr;
    GK_TRY(get_cache(M, &C));
    GridPlan P;
    GK_TRY(grid_plan(M, C, m + 1, &P));
    P.half = P.R <= GRID_GM_HALF_ROWS && P.R * M->K <= GRID_GM_HALF_ENTRIES &&
             (int64_t)grid_gm_smem<GRID_HALF, V, T>(false, m, P.R, M->K) <= P.room[1];
    auto smem_of = [&](bool st) {
        return P.half ? grid_gm_smem<GRID_HALF, V, T>(st, m, P.R, M->K)
                      : grid_gm_smem<GRID_FULL, V, T>(st, m, P.R, M->K);
    };
    const int64_t room = P.room[P.half ? 1 : 0];
    const bool staged = (int64_t)smem_of(true) <= room;
    const size_t smem = smem_of(staged);
    const size_t vbytes = ((size_t)P.nb * P.R * sizeof(T) + 255) & ~(size_t)255;
    if ((int64_t)smem > room) return GK_ERR_UNSUPPORTED;
    const bool prec = pkind == 1;
    if (prec) GK_TRY(ensure_jacobi(M, s));
    GK_TRY(grid_vectors(C, vbytes * (size_t)(m + 3)));
    char* v = static_cast<char*>(C->gvecs.ptr);
    GridGmArgs<V, T> a;
    a.n = n;
    a.R = (int32_t)P.R;
    a.K = M->K;
    a.m = m;
    a.stride = M->stride;
    a.col = M->col;
    a.val = (const V*)M->val;
    a.b = b;
    a.x0 = x;
    a.p = (T*)v;
    a.x = (T*)(v + vbytes);
    a.basis = (T*)(v + 2 * vbytes);
    a.ldv = (int64_t)(vbytes / sizeof(T));
    a.dinv = prec ? (const T*)M->dinv : nullptr;
    a.slots = P.slots();
    a.arrived = P.arrived();
    a.err = P.err();
    a.out = P.out();
    a.tol = tol;
    a.max_iters = max_iters;
    a.stag = inner ? 0.95 : 0.0;
    a.wait_ns = M->wait_ns;
    a.between = grid_polls_between(a.wait_ns);
    auto go = [&](auto nt, auto st) -> gk_status {
        constexpr int NT = decltype(nt)::value;
        constexpr bool ST = decltype(st)::value;
        return prec ? grid_launch<NT>(k_grid_gmres<NT, V, T, ST, true>, a, P, smem, s)
                    : grid_launch<NT>(k_grid_gmres<NT, V, T, ST, false>, a, P, smem, s);
    };
    auto go_staged = [&](auto nt) -> gk_status {
        return staged ? go(nt, std::true_type{}) : go(nt, std::false_type{});
    };
    return grid_run(C, P, s, out, n, a.x, x, [&]() -> gk_status {
        return P.half ? go_staged(std::integral_constant<int, GRID_HALF>{})
                      : go_staged(std::integral_constant<int, GRID_FULL>{});
    });
}

extern template gk_status solve_grid_gmres<double, double>(gk_matrix, const double*, double*, int,
                                                           double, int32_t, int, cudaStream_t,
                                                           SolveOut*, bool);
extern template gk_status solve_grid_gmres<float, float>(gk_matrix, const float*, float*, int,
                                                         double, int32_t, int, cudaStream_t,
                                                         SolveOut*, bool);
extern template gk_status solve_grid_gmres<__nv_bfloat16, float>(gk_matrix, const float*, float*,
                                                                 int, double, int32_t, int,
                                                                 cudaStream_t, SolveOut*, bool);
extern template gk_status solve_grid_gmres<__half, float>(gk_matrix, const float*, float*, int,
                                                          double, int32_t, int, cudaStream_t,
                                                          SolveOut*, bool);

}  // namespace gk
