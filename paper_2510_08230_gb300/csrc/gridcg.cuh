// gridcg.cuh - CG (none or Jacobi) as one persistent cooperative kernel over
// the whole GPU, for matrices whose solver layout is ELL.
//
// Why: the multi-kernel engine spends a fixed ~9 us per reducing kernel on
// the grid reduction's tail (fence, ticket, the last block's pass over the
// partials, the next launch) while the other SMs idle.  Per Jacobi-CG
// iteration, multi-kernel against this kernel (GB300, us; the FP64 pipe's
// own floor in brackets): 17,030-row 2D stencil 20.0 / 7.9, 117,453-row 3D
// stencil 22.3 / 11.4 (2.6), 10^6-row 3D stencil 59.9 / 37.7 (22), 128^3
// diffusion 98 / 69.5 (47), in FP32 56 / 30; 121 entries a row, n = 30,000:
// 75.6 / 24.3, n = 500,000: 316 / 175.  Six solves at once, 600 iterations
// each, in ms: 17K to 25K rows 25.5 / 12.1 (alone, in turn: 74 / 30), 70K to
// 430K rows in FP64 38 / 43 to 52 (97 / 58), in FP32 24.6 / 24 to 31 (79 / 40):
// there two grids fill the GPU and the others queue, which the multi-kernel
// engine's kernels do not.  What is left on small matrices is latency: the
// block's FP64 tree (~2,300 cycles a reduction), the hand-offs (~1,700 to 2,600
// each) and FP64 divisions; on large ones the FP64 pipe (128^3: 97,000 of
// 153,000 cycles).
//
// Block k owns rows [kR, (k+1)R).  The vectors only their owner reads
// (r, q, and x and the inverse diagonal when they fit) stay in its shared
// memory for the whole solve, small matrices with them; only the gathered
// vector p goes through global memory.  Per iteration (Hestenes-Stiefel, the
// recurrence and the per-row arithmetic of the multi-kernel engine) three
// grid-wide hand-offs (gridbase.cuh): <p, q>; <r, z> and ||r||^2; p published.
#pragma once

#include "gridbase.cuh"

namespace gk {

template <typename V, typename T>
struct GridCgArgs {
    int32_t n, R, K;
    int64_t stride;
    const int32_t* col;
    const V* val;
    const T* b;
    const T* x0;   // the initial guess
    T* x;          // the solution, padded to whole blocks; mode 2 works on it
    const T* dinv; // null: no preconditioner
    T* p;          // gathered vector, padded to whole blocks
    unsigned long long *slots, *arrived;
    int32_t* err;
    GridOut* out;
    double tol;
    int32_t max_iters, inner, stall;
    uint64_t wait_ns;
    unsigned between;  // see GridTeam
};

// Shared-memory modes: what a block keeps there beside r and q.
//   0: x, the inverse diagonal and its rows of the matrix
//   1: x and the inverse diagonal
//   2: nothing more
template <int NT, typename V, typename T>
size_t grid_cg_smem(int mode, int64_t R, int64_t K) {
    size_t s = GRID_RED<NT> + (size_t)R * sizeof(T) * (mode == 2 ? 2 : 4);
    if (mode == 0) s += (size_t)(R * K) * (sizeof(V) + 4);
    return s;
}

template <int NT, typename V, typename T, int MODE, bool PREC>
__global__ void __launch_bounds__(NT, GRID_FULL / NT) k_grid_cg(const GridCgArgs<V, T> A) {
    extern __shared__ __align__(128) unsigned char smem[];
    T* rs = reinterpret_cast<T*>(smem + GRID_RED<NT>);
    const int32_t R = A.R;
    T* qs = rs + R;               // q, and z after the update
    T* xs = qs + R;               // modes 0 and 1
    T* ds = xs + R;
    V* s_val = reinterpret_cast<V*>(ds + R);
    __shared__ double part[8];
    __shared__ int s_code;
    // the solve's scalars, kept by the lane that runs the sums' fins
    __shared__ struct {
        double bn, thr, thr2, tn, rec2, best2, rho, alpha, beta;
    } S;
    const int tid = threadIdx.x;
    const int32_t r0 = (int32_t)blockIdx.x * R;
    const int32_t nloc = min(R, A.n - r0);  // >= 1
    GridTeam<NT> team{A.slots, A.arrived, A.err, A.wait_ns, A.between, (int)gridDim.x, 0, nloc > NT / 2,
                  reinterpret_cast<double*>(smem), part, &s_code, 0u};
    const GridRows<NT, V, T, MODE == 0> rows{R, A.K, r0, nloc, A.stride, A.col, A.val, s_val,
                                             reinterpret_cast<int32_t*>(s_val + (size_t)(MODE == 0 ? R * A.K : 0))};
    rows.stage();
    for (int32_t li = tid; li < nloc; li += NT) {
        const T xi = A.x0[r0 + li];
        if constexpr (MODE != 2) {
            xs[li] = xi;
            ds[li] = PREC ? A.dinv[r0 + li] : T(0);
        } else {
            A.x[r0 + li] = xi;
        }
        A.p[r0 + li] = xi;
    }

    auto dinv_at = [&](int32_t li) -> T {
        if constexpr (MODE != 2) return ds[li];
        else return A.dinv[r0 + li];
    };

    // r = b - A x for the x published in A.p.  The first one also takes
    // ||b||; its code: 0 go on, else why the solve ends here.
    auto residual = [&](bool first) -> int {
        T a[2] = {T(0), T(0)};
        rows.product(A.p, [&](int32_t li, T s) {
            const T bi = A.b[r0 + li];
            const T ri = bi - s;
            rs[li] = ri;
            a[0] = fmadd(bi, bi, a[0]);
            a[1] = fmadd(ri, ri, a[1]);
        });
        const double v[2] = {(double)a[0], (double)a[1]};
        return team.sum<2>(0, v, [&](const double* t) -> int {
            if (first) {
                S.bn = sqrt(t[0]);
                S.thr = A.tol * S.bn;
                S.thr2 = S.thr * S.thr;
                S.rec2 = t[1];
                S.best2 = 0.0;
            }
            S.tn = sqrt(t[1]);
            if (!isfinite(S.bn) || (S.bn > 0.0 && !isfinite(S.tn))) return END_NAN;
            return S.bn == 0.0 ? END_ZERO : S.tn <= S.thr ? END_OK : 0;
        });
    };
    // z = M^-1 r ; p = z ; rho = <r, z>, published
    auto start = [&]() -> bool {
        T a = T(0);
        rows.each([&](int32_t li) {
            const T ri = rs[li];
            const T zi = PREC ? dinv_at(li) * ri : ri;
            A.p[r0 + li] = zi;
            a = fmadd(ri, zi, a);
        });
        const double v[1] = {(double)a};
        return team.sum<1>(1, v, [&](const double* t) {
                   S.rho = t[0];
                   return 0;
               }) == 0 && team.publish();
    };
    // x into A.p, published
    auto publish_x = [&]() -> bool {
        rows.each([&](int32_t li) { A.p[r0 + li] = MODE != 2 ? xs[li] : A.x[r0 + li]; });
        return team.publish();
    };

    int iters = 0, restarts = 0, best_iter = 0;
    int end = team.publish() ? residual(true) : END_TIMEOUT;
    bool changed = false;  // x has changed since S.tn was taken
    if (end == 0 && !start()) end = END_TIMEOUT;
    while (end == 0) {
        // q = A p ; <p, q>
        T apq = T(0);
        rows.product(A.p, [&](int32_t li, T s) {
            qs[li] = s;
            apq = fmadd(A.p[r0 + li], s, apq);
        });
        const double vpq[1] = {(double)apq};
        end = team.sum<1>(0, vpq, [&](const double* t) -> int {
            S.alpha = S.rho / t[0];
            return !isfinite(t[0]) ? END_NAN : t[0] <= 0.0 ? END_BREAKDOWN : 0;
        });
        if (end != 0) break;
        // x += alpha p ; r -= alpha q ; z = M^-1 r ; <r, z>, <r, r>
        T a[2] = {T(0), T(0)};
        {
            const T alpha = (T)S.alpha;
            rows.each([&](int32_t li) {
                const T pi = A.p[r0 + li];
                if constexpr (MODE != 2) xs[li] = fmadd(alpha, pi, xs[li]);
                else A.x[r0 + li] = fmadd(alpha, pi, A.x[r0 + li]);
                const T ri = fmadd(-alpha, qs[li], rs[li]);
                rs[li] = ri;
                if constexpr (PREC) {
                    const T zi = dinv_at(li) * ri;
                    qs[li] = zi;
                    a[1] = fmadd(ri, zi, a[1]);
                }
                a[0] = fmadd(ri, ri, a[0]);
            });
        }
        changed = true;
        ++iters;
        const double v[2] = {(double)a[0], (double)a[1]};
        end = team.sum<PREC ? 2 : 1>(1, v, [&](const double* t) -> int {
            const double rr = t[0], rz = t[PREC ? 1 : 0];
            S.rec2 = rr;
            if (!isfinite(rr) || !isfinite(rz)) return END_NAN;
            if (rr <= S.thr2) return PASSED;
            if (iters >= A.max_iters) return END_CAP;
            if (A.stall > 0) {  // no 10 % gain on the best residual for `stall` iterations
                if (!(S.best2 > 0.0) || rr < 0.81 * S.best2) {
                    S.best2 = rr;
                    best_iter = iters;
                } else if (iters - best_iter >= A.stall) {
                    return END_CAP;
                }
            }
            S.beta = rz / S.rho;
            S.rho = rz;
            return 0;
        });
        if (end == PASSED) {
            // the recurrence residual passes: the true residual decides, and
            // on failure replaces r; a refinement's inner solve stops after
            // two replacements
            if (A.inner && restarts >= 2) {
                end = END_INNER;
                break;
            }
            end = publish_x() ? residual(false) : END_TIMEOUT;
            changed = false;
            if (end == 0 && iters >= A.max_iters) end = END_CAP;
            if (end != 0) break;
            restarts += 1;
            if (!start()) end = END_TIMEOUT;
            continue;
        }
        if (end != 0) break;
        const T beta = (T)S.beta;
        rows.each([&](int32_t li) {
            const T zi = PREC ? qs[li] : rs[li];
            A.p[r0 + li] = fmadd(beta, A.p[r0 + li], zi);
        });
        rows.prefetch_first();  // the next product's first rows
        if (!team.publish()) end = END_TIMEOUT;
    }
    if (changed && (end == END_NAN || end == END_BREAKDOWN || end == END_CAP))
        if (!publish_x() || residual(false) == END_TIMEOUT) end = END_TIMEOUT;
    for (int32_t li = tid; li < nloc; li += NT) {
        if (end == END_ZERO) A.x[r0 + li] = T(0);
        else if constexpr (MODE != 2) A.x[r0 + li] = xs[li];
    }
    if (blockIdx.x == 0 && tid == 0) {
        GridOut o;
        o.status = end_status(end);
        o.iters = iters;
        o.restarts = restarts;
        o.pad = 0;
        o.rec = S.bn > 0.0 ? sqrt(S.rec2) / S.bn : 0.0;
        o.tru = end == END_INNER ? o.rec : S.bn > 0.0 ? S.tn / S.bn : 0.0;
        *A.out = o;
    }
}

// ------------------------------------------------------------ host side

// One CG solve on k_grid_cg.  GK_ERR_UNSUPPORTED, with x untouched: the matrix
// is too large for the blocks' shared memory, there is no room for the
// vectors, the grid cannot be resident at once, or a wait ran out.
template <typename V, typename T>
gk_status solve_grid_cg(gk_matrix M, const T* b, T* x, int pkind, double tol, int32_t max_iters,
                        cudaStream_t s, SolveOut* out, bool inner) {
    const int32_t n = M->n;
    SolverCache* C = nullptr;
    GK_TRY(get_cache(M, &C));
    GridPlan P;
    GK_TRY(grid_plan(M, C, 0, &P));
    int mode = 0;
    while (mode < 2 && (int64_t)grid_cg_smem<GRID_HALF, V, T>(mode, P.R, M->K) > P.room[1]) ++mode;
    P.half = mode < 2;
    if (!P.half) {
        mode = 0;
        while (mode < 3 && (int64_t)grid_cg_smem<GRID_FULL, V, T>(mode, P.R, M->K) > P.room[0]) ++mode;
        if (mode == 3) return GK_ERR_UNSUPPORTED;
    }
    const bool prec = pkind == 1;
    if (prec) GK_TRY(ensure_jacobi(M, s));
    const size_t vbytes = ((size_t)P.nb * P.R * sizeof(T) + 255) & ~(size_t)255;
    GK_TRY(grid_vectors(C, vbytes * 2));
    GridCgArgs<V, T> a;
    a.n = n;
    a.R = (int32_t)P.R;
    a.K = M->K;
    a.stride = M->stride;
    a.col = M->col;
    a.val = (const V*)M->val;
    a.b = b;
    a.x0 = x;
    a.x = (T*)(static_cast<char*>(C->gvecs.ptr) + vbytes);
    a.dinv = prec ? (const T*)M->dinv : nullptr;
    a.p = (T*)C->gvecs.ptr;
    a.slots = P.slots();
    a.arrived = P.arrived();
    a.err = P.err();
    a.out = P.out();
    a.tol = tol;
    a.max_iters = max_iters;
    a.inner = inner ? 1 : 0;
    a.stall = inner ? 200 : 0;
    a.wait_ns = M->wait_ns;
    a.between = grid_polls_between(a.wait_ns);
    auto go = [&](auto nt, auto md) -> gk_status {
        constexpr int NT = decltype(nt)::value, MD = decltype(md)::value;
        const size_t smem = grid_cg_smem<NT, V, T>(MD, P.R, M->K);
        return prec ? grid_launch<NT>(k_grid_cg<NT, V, T, MD, true>, a, P, smem, s)
                    : grid_launch<NT>(k_grid_cg<NT, V, T, MD, false>, a, P, smem, s);
    };
    constexpr std::integral_constant<int, GRID_FULL> full;
    constexpr std::integral_constant<int, GRID_HALF> half;
    constexpr std::integral_constant<int, 0> m0;
    constexpr std::integral_constant<int, 1> m1;
    constexpr std::integral_constant<int, 2> m2;
    return grid_run(C, P, s, out, n, a.x, x, [&]() -> gk_status {
        return P.half      ? (mode == 0 ? go(half, m0) : go(half, m1))
               : mode == 0 ? go(full, m0)
               : mode == 1 ? go(full, m1)
                           : go(full, m2);
    });
}

extern template gk_status solve_grid_cg<double, double>(gk_matrix, const double*, double*, int,
                                                        double, int32_t, cudaStream_t, SolveOut*,
                                                        bool);
extern template gk_status solve_grid_cg<float, float>(gk_matrix, const float*, float*, int, double,
                                                      int32_t, cudaStream_t, SolveOut*, bool);
extern template gk_status solve_grid_cg<__nv_bfloat16, float>(gk_matrix, const float*, float*, int,
                                                              double, int32_t, cudaStream_t,
                                                              SolveOut*, bool);
extern template gk_status solve_grid_cg<__half, float>(gk_matrix, const float*, float*, int, double,
                                                       int32_t, cudaStream_t, SolveOut*, bool);

}  // namespace gk
