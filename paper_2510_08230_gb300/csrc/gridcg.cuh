// gridcg.cuh - CG (none or Jacobi) as one persistent cooperative kernel over
// the whole GPU, for matrices whose solver layout is ELL.
//
// Why: the multi-kernel engine spends a fixed ~9 us per reducing kernel on
// the grid reduction's tail (fence, ticket, the last block's pass over the
// partials, the next launch) while the other SMs idle.  Per Jacobi-CG
// iteration, multi-kernel against this kernel (GB300, us; the FP64 pipe's
// own floor in brackets): 17,030-row 2D stencil 20.0 / 9.4, 117,453-row 3D
// stencil 22.3 / 12.4 (2.6), 10^6-row 3D stencil 59.9 / 39.3 (22), 128^3
// diffusion 98 / 72 (47), in FP32 57 / 32; 121 entries a row, n = 30,000:
// 75.6 / 25.4.  Six serving-size solves at once: 115 ms / 98 ms.  What is
// left on small matrices is latency: the block's FP64 tree (~2,300 cycles a
// reduction), the hand-offs (~1,700 to 2,600 each) and FP64 divisions; on
// large ones the FP64 pipe (128^3: 97,000 of 153,000 cycles).
//
// Block k owns rows [kR, (k+1)R).  The vectors only their owner reads
// (r, q, and x and the inverse diagonal when they fit) stay in its shared
// memory for the whole solve, small matrices with them; only the gathered
// vector p goes through global memory.  Per iteration (Hestenes-Stiefel, the
// recurrence and the per-row arithmetic of the multi-kernel engine) three
// grid-wide hand-offs: <p, q>; <r, z> and ||r||^2; p published.
//
// Hand-off of a reduction: every block posts its partial sums to slots of
// its own, and warp 0 of every block polls all slots (at most 5 per lane,
// loaded together), adds them in one fixed order and forms the scalars, so
// all blocks take identical decisions and results do not depend on timing.
// A slot holding SLOT_EMPTY has not been posted yet: value and signal travel
// in one 8-byte exchange, and no fence is needed because no data is handed
// over with it.  Measured on 152 blocks, cycles from post to all seen:
// exchange 1,700, relaxed store 2,000 to 2,700, a master block that collects
// and rebroadcasts 4,500, clusters of 8 or 16 with one poller each 4,400;
// with a release fence (p published): a counter 2,500, stores 4,300.
// Slots come in three rounds (one round an iteration); a block empties its
// slots of round k + 1 before it publishes p in round k: by then every block
// has left round k - 2, which used them.  Every poll is bounded.
#pragma once

#include "solve_engine.cuh"

namespace gk {

constexpr unsigned long long SLOT_EMPTY = ~0ull;
constexpr int GCG_POLLS = 5;                   // slots per polling lane
constexpr int GCG_MAX_BLOCKS = 32 * GCG_POLLS;
constexpr int GCG_VALUES = 4;                  // slots a block and round: 2 sums of up to 2 values
constexpr int GCG_ROUNDS = 3;

// why a solve ends (0: it goes on); PASSED: its recurrence residual passed
enum : int { END_OK = 1, END_ZERO, END_INNER, END_CAP, END_NAN, END_BREAKDOWN, END_TIMEOUT, PASSED };

struct GridCgOut {
    int32_t status, iters, restarts, pad;
    double rec, tru;
};

template <typename V, typename T>
struct GridCgArgs {
    int32_t n, R, K;
    int64_t stride;
    const int32_t* col;
    const V* val;
    const T* b;
    const T* x0;   // the initial guess
    T* x;          // the solution; mode 2 works on it (16-byte aligned, padded to whole blocks)
    const T* dinv; // null: no preconditioner
    T* p;          // gathered vector, padded to whole blocks
    unsigned long long* slots;  // [GCG_ROUNDS][GCG_VALUES][gridDim.x], SLOT_EMPTY at launch
    unsigned long long* arrived;  // blocks that have published, all rounds (0 at launch)
    int32_t* err;
    GridCgOut* out;
    double tol;
    int32_t max_iters, inner, stall;
    uint64_t wait_ns;
};

// Shared-memory modes: what a block keeps there beside r and q.
//   0: x, the inverse diagonal and its rows of the matrix
//   1: x and the inverse diagonal
//   2: nothing more
// One row per thread and pass: with 32 warps an SM's FP64 pipe (a warp
// instruction per 16 cycles) always finds one whose loads have landed.
constexpr int GCG_NT = 1024;
constexpr size_t GCG_RED = 2 * (GCG_NT / 2) * sizeof(double);

template <typename V, typename T>
size_t grid_cg_smem(int mode, int64_t R, int64_t K) {
    size_t s = GCG_RED + (size_t)R * sizeof(T) * (mode == 2 ? 2 : 4);
    if (mode == 0) s += (size_t)(R * K) * (sizeof(V) + 4);
    return s;
}

__device__ __forceinline__ unsigned long long ld_slot(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
// Sums a and b over the warp together: a in lanes 0 to 15, b in lanes 16 to
// 31 (five adds instead of ten).
__device__ __forceinline__ double warp_sum2(double a, double b) {
    const bool low = (threadIdx.x & 16) == 0;
    double t = (low ? a : b) + __shfl_xor_sync(0xffffffffu, low ? b : a, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

template <typename V, typename T, int MODE, bool PREC>
__global__ void __launch_bounds__(GCG_NT, 1) k_grid_cg(const GridCgArgs<V, T> A) {
    constexpr int NT = GCG_NT, HT = NT / 2;
    constexpr int CH = 8;  // entries of a row in flight
    extern __shared__ __align__(128) unsigned char smem[];
    double* red = reinterpret_cast<double*>(smem);
    T* rs = reinterpret_cast<T*>(smem + GCG_RED);
    const int32_t R = A.R;
    T* qs = rs + R;               // q, and z after the update
    T* xs = qs + R;               // modes 0 and 1
    T* ds = xs + R;
    V* ms_val = reinterpret_cast<V*>(ds + R);  // mode 0: entry j of row li at j R + li
    int32_t* ms_col = reinterpret_cast<int32_t*>(ms_val + (size_t)(MODE == 0 ? R * A.K : 0));
    __shared__ double part[8];    // sums of 128 threads' values
    // the solve's scalars, kept by lane 0 of the polling warp, and its decision
    __shared__ struct {
        double bn, thr, thr2, tn, rec2, best2, rho, alpha, beta;
    } S;
    __shared__ int s_code;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nb = (int)gridDim.x;
    const int32_t r0 = (int32_t)blockIdx.x * R;
    const int32_t nloc = min(R, A.n - r0);  // >= 1
    unsigned round = 0;
    auto slot = [&](unsigned rd, int v) { return A.slots + ((size_t)(rd % GCG_ROUNDS) * GCG_VALUES + v) * nb; };

    // Warp 0 spins until ready() holds in all lanes; false: the budget ran
    // out, here or in another block.
    auto wait = [&](auto&& ready) -> bool {
        uint64_t t0 = 0;
        for (unsigned spin = 0;; ++spin) {
            if (__all_sync(0xffffffffu, ready())) return true;
            if ((spin & 255u) != 255u) continue;
            bool stop = false;
            if (lane == 0) {
                const uint64_t t = globaltimer_ns();
                if (t0 == 0) t0 = t;
                stop = t - t0 > A.wait_ns || *reinterpret_cast<volatile int32_t*>(A.err) != 0;
                if (stop) atomicExch(A.err, 1);
            }
            if (__any_sync(0xffffffffu, stop)) return false;
        }
    };

    // Sums NA values over the grid, runs fin(totals) on one lane (which leaves
    // scalars in S and a code) and returns the code in every thread.  kind 0 and 1: each at most once a round.  A warp's FP64
    // instruction holds its sub-partition's pipe for 65 cycles whatever its
    // mask, so the block's tree is spread over the four sub-partitions: one
    // add for the upper half of the threads, then four warps add four values
    // a lane and shuffle.
    auto grid_sum = [&](auto na, int kind, const double* v, auto&& fin) -> int {
        constexpr int NA = decltype(na)::value;
        const bool upper = nloc > HT;  // otherwise the upper half holds zeros
        if (upper) {
            if (tid >= HT)
#pragma unroll
                for (int a = 0; a < NA; ++a) red[a * HT + tid - HT] = v[a];
            __syncthreads();
        }
        if (tid < HT)
#pragma unroll
            for (int a = 0; a < NA; ++a) red[a * HT + tid] = upper ? v[a] + red[a * HT + tid] : v[a];
        __syncthreads();
        if (warp < 4) {
            const double* w = red + warp * 128 + lane;
            const double t0 = (w[0] + w[32]) + (w[64] + w[96]);
            if constexpr (NA == 2) {
                w += HT;
                const double t = warp_sum2(t0, (w[0] + w[32]) + (w[64] + w[96]));
                if ((lane & 15) == 0) part[(lane >> 2) + warp] = t;
            } else {
                const double t = warp_sum(t0);
                if (lane == 0) part[warp] = t;
            }
        }
        __syncthreads();
        if (warp == 0) {
            if (lane < NA) {
                const double* w = part + 4 * lane;
                unsigned long long u =
                    (unsigned long long)__double_as_longlong((w[0] + w[1]) + (w[2] + w[3]));
                if (u == SLOT_EMPTY) u = 0x7ff8000000000000ull;  // any other NaN
                atomicExch(slot(round, 2 * kind + lane) + blockIdx.x, u);
            }
            const unsigned long long* sl = slot(round, 2 * kind);
            unsigned long long u[NA][GCG_POLLS];
            const bool ok = wait([&] {
                bool all = true;
#pragma unroll
                for (int a = 0; a < NA; ++a)
#pragma unroll
                    for (int j = 0; j < GCG_POLLS; ++j) {
                        const int i = lane + 32 * j;
                        u[a][j] = i < nb ? ld_slot(sl + (size_t)a * nb + i) : 0ull;
                    }
#pragma unroll
                for (int a = 0; a < NA; ++a)
#pragma unroll
                    for (int j = 0; j < GCG_POLLS; ++j) all &= u[a][j] != SLOT_EMPTY;
                return all;
            });
            double tot[NA];
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                double x[GCG_POLLS];
#pragma unroll
                for (int j = 0; j < GCG_POLLS; ++j) x[j] = __longlong_as_double((long long)u[a][j]);
                tot[a] = ((x[0] + x[1]) + (x[2] + x[3])) + x[4];
            }
            if constexpr (NA == 2) {
                tot[0] = warp_sum2(tot[0], tot[1]);
                tot[1] = __shfl_sync(0xffffffffu, tot[0], 16);
            } else {
                tot[0] = warp_sum(tot[0]);
            }
            if (lane == 0) s_code = ok ? fin(tot) : END_TIMEOUT;
        }
        __syncthreads();
        return s_code;
    };
    static_assert(GCG_POLLS == 5, "grid_sum adds five polled values a lane");

    // Ends a round: everything this block wrote to A.p is visible to every
    // block afterwards.  False: a wait ran out.
    auto publish = [&]() -> bool {
        if (tid < GCG_VALUES) *(slot(round + 1, tid) + blockIdx.x) = SLOT_EMPTY;
        __syncthreads();
        ++round;
        if (warp == 0) {
            if (lane == 0) {
                __threadfence();
                atomicAdd(A.arrived, 1ull);
            }
            const unsigned long long want = (unsigned long long)round * nb;
            const bool ok = wait([&] { return lane != 0 || ld_slot(A.arrived) >= want; });
            __threadfence();
            if (lane == 0) s_code = ok ? 0 : -1;
        }
        __syncthreads();
        return s_code == 0;
    };

    // ---- setup: the block's rows and vectors
    if constexpr (MODE == 0) {
        for (int32_t j = 0; j < A.K; ++j)
            for (int32_t li = tid; li < nloc; li += NT) {
                ms_val[j * R + li] = A.val[(int64_t)j * A.stride + r0 + li];
                ms_col[j * R + li] = A.col[(int64_t)j * A.stride + r0 + li];
            }
    }
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

    // f(li) for every row of this thread (the same rows each time)
    auto rows = [&](auto&& f) {
#pragma unroll 2
        for (int32_t li = tid; li < nloc; li += NT) f(li);
    };
    // Modes 1 and 2: brings the matrix entries of the 32 rows from li on (a
    // multiple of 32) into L2 while the warp works on others: one lane per
    // 128-byte line, so it costs an instruction or two and no registers.
    auto prefetch = [&](int32_t li) {
        constexpr int VL = 32 * (int)sizeof(V) > 128 ? 32 * (int)sizeof(V) / 128 : 1;
        if (li >= nloc) return;
        const uint32_t row = (uint32_t)(r0 + li);
        for (int k = lane; k < A.K * (VL + 1); k += 32) {
            const uint32_t j = (uint32_t)k / (VL + 1), l = (uint32_t)k % (VL + 1);
            const uint32_t at = j * (uint32_t)A.stride + row;
            const char* q = l == VL ? reinterpret_cast<const char*>(A.col) + at * 4u
                                    : reinterpret_cast<const char*>(A.val) + at * (uint32_t)sizeof(V) + 128u * l;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(q));
        }
    };
    // f(li, sum): the row times the gathered vector (plain loads: p changes
    // between rounds, and the fences of publish() order them).  Offsets into
    // the matrix are 32-bit bytes (the host checks that they fit).
    auto spmv = [&](auto&& f) {
        const T* p = A.p;
        const uint32_t ld = MODE == 0 ? (uint32_t)R : (uint32_t)A.stride;
        const char* vals = reinterpret_cast<const char*>(MODE == 0 ? ms_val : A.val);
        const char* cols = reinterpret_cast<const char*>(MODE == 0 ? ms_col : A.col);
        for (int32_t li = tid; li < nloc; li += NT) {
            if constexpr (MODE != 0) prefetch(li - lane + NT);
            T s = T(0);
            uint32_t at = MODE == 0 ? (uint32_t)li : (uint32_t)(r0 + li);
            for (int32_t left = A.K; left > 0; left -= CH, at += CH * ld) {
                int32_t c[CH];
                V v[CH];
                T xv[CH];
#pragma unroll
                for (int u = 0; u < CH; ++u) {
                    c[u] = -1;
                    if (u < left) {
                        const int32_t* q = reinterpret_cast<const int32_t*>(cols + (at + u * ld) * 4u);
                        c[u] = MODE == 0 ? *q : __ldcs(q);
                    }
                }
#pragma unroll
                for (int u = 0; u < CH; ++u)
                    if (u < left)
                        v[u] = *reinterpret_cast<const V*>(vals + (at + u * ld) * (uint32_t)sizeof(V));
#pragma unroll
                for (int u = 0; u < CH; ++u) xv[u] = c[u] >= 0 ? p[c[u]] : T(0);
#pragma unroll
                for (int u = 0; u < CH; ++u)
                    if (u < left) s = fmadd(cvt<T>(v[u]), xv[u], s);
            }
            f(li, s);
        }
    };
    auto dinv_at = [&](int32_t li) -> T {
        if constexpr (MODE != 2) return ds[li];
        else return A.dinv[r0 + li];
    };
    using one = std::integral_constant<int, 1>;
    using two = std::integral_constant<int, 2>;

    // r = b - A x for the x published in A.p.  The first one also takes
    // ||b||; its code: 0 go on, else why the solve ends here.
    auto residual = [&](bool first) -> int {
        T a[2] = {T(0), T(0)};
        spmv([&](int32_t li, T s) {
            const T bi = A.b[r0 + li];
            const T ri = bi - s;
            rs[li] = ri;
            a[0] = fmadd(bi, bi, a[0]);
            a[1] = fmadd(ri, ri, a[1]);
        });
        const double v[2] = {(double)a[0], (double)a[1]};
        return grid_sum(two{}, 0, v, [&](const double* t) -> int {
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
        rows([&](int32_t li) {
            const T ri = rs[li];
            const T zi = PREC ? dinv_at(li) * ri : ri;
            A.p[r0 + li] = zi;
            a = fmadd(ri, zi, a);
        });
        const double v[1] = {(double)a};
        return grid_sum(one{}, 1, v, [&](const double* t) {
                   S.rho = t[0];
                   return 0;
               }) >= 0 && publish();
    };
    // x into A.p, published
    auto publish_x = [&]() -> bool {
        rows([&](int32_t li) { A.p[r0 + li] = MODE != 2 ? xs[li] : A.x[r0 + li]; });
        return publish();
    };

    int iters = 0, restarts = 0, best_iter = 0;
    int end = publish() ? residual(true) : END_TIMEOUT;
    bool changed = false;  // x has changed since S.tn was taken
    if (end == 0 && !start()) end = END_TIMEOUT;
    while (end == 0) {
        // q = A p ; <p, q>
        T apq = T(0);
        spmv([&](int32_t li, T s) {
            qs[li] = s;
            apq = fmadd(A.p[r0 + li], s, apq);
        });
        const double vpq[1] = {(double)apq};
        end = grid_sum(one{}, 0, vpq, [&](const double* t) -> int {
            S.alpha = S.rho / t[0];
            return !isfinite(t[0]) ? END_NAN : t[0] <= 0.0 ? END_BREAKDOWN : 0;
        });
        if (end != 0) break;
        // x += alpha p ; r -= alpha q ; z = M^-1 r ; <r, z>, <r, r>
        T a[2] = {T(0), T(0)};
        {
            const T alpha = (T)S.alpha;
            rows([&](int32_t li) {
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
        end = grid_sum(std::integral_constant<int, PREC ? 2 : 1>{}, 1, v, [&](const double* t) -> int {
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
        rows([&](int32_t li) {
            const T zi = PREC ? qs[li] : rs[li];
            A.p[r0 + li] = fmadd(beta, A.p[r0 + li], zi);
        });
        if constexpr (MODE != 0) prefetch(tid - lane);  // the next product's first rows
        if (!publish()) end = END_TIMEOUT;
    }
    if (changed && (end == END_NAN || end == END_BREAKDOWN || end == END_CAP))
        if (!publish_x() || residual(false) == END_TIMEOUT) end = END_TIMEOUT;
    for (int32_t li = tid; li < nloc; li += NT) {
        if (end == END_ZERO) A.x[r0 + li] = T(0);
        else if constexpr (MODE != 2) A.x[r0 + li] = xs[li];
    }
    if (blockIdx.x == 0 && tid == 0) {
        GridCgOut o;
        o.status = end == END_OK || end == END_ZERO || end == END_INNER ? GK_OK
                   : end == END_NAN                                     ? GK_ERR_NAN
                   : end == END_BREAKDOWN                               ? GK_BREAKDOWN
                   : end == END_CAP                                     ? GK_NOT_CONVERGED
                                                                        : GK_ERR_TIMEOUT;
        o.iters = iters;
        o.restarts = restarts;
        o.pad = 0;
        o.rec = S.bn > 0.0 ? sqrt(S.rec2) / S.bn : 0.0;
        o.tru = end == END_INNER ? o.rec : S.bn > 0.0 ? S.tn / S.bn : 0.0;
        *A.out = o;
    }
}

// ------------------------------------------------------------ host side

// Cooperative grids of this process run one at a time (each fills the GPU's
// shared memory): the holder's stream is drained first, so the lock is held
// for the solve alone.
std::mutex& grid_cg_mutex();

// Whether gk_solve's automatic engine may take this solve to k_grid_cg.
inline bool grid_cg_admits(gk_matrix M, int method, int pkind) {
    return method == GK_CG && pkind <= 1 && M->fmt == GK_ELL && M->K > 0 &&
           !getenv("GK_SOLVE_UNROLLED") && !solve_loop_on_host();
}

// One CG solve on k_grid_cg.  GK_ERR_UNSUPPORTED: the matrix is too large
// for the blocks' shared memory, or the grid cannot be resident at once.
template <typename V, typename T>
gk_status solve_grid_cg(gk_matrix M, const T* b, T* x, int pkind, double tol, int32_t max_iters,
                        cudaStream_t s, SolveOut* out, bool inner) {
    const int32_t n = M->n;
    const int sms = std::min(num_sms(), GCG_MAX_BLOCKS);
    const int64_t R = (((int64_t)n + sms - 1) / sms + 63) / 64 * 64;
    const int nb = (int)(((int64_t)n + R - 1) / R);
    int dev = 0, optin = 0, coop = 0;
    GK_CUDA(cudaGetDevice(&dev));
    GK_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    GK_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    const int64_t room = (int64_t)optin - 1024;  // the kernels' static shared memory
    int mode = 0;
    while (mode < 3 && (int64_t)grid_cg_smem<V, T>(mode, R, M->K) > room) ++mode;
    if (mode == 3) return GK_ERR_UNSUPPORTED;
    if (!coop) return GK_ERR_UNSUPPORTED;
    // the kernel's byte offsets into the matrix have 32 bits (a chunk of 8
    // entries past the last is formed, not read)
    if ((uint64_t)(M->K + 8) * (uint64_t)M->stride * sizeof(V) >= (1ull << 32)) return GK_ERR_UNSUPPORTED;
    const bool prec = pkind == 1;
    if (prec) GK_TRY(ensure_jacobi(M, s));
    SolverCache* C = nullptr;
    GK_TRY(get_cache(M, &C));
    const size_t vbytes = ((size_t)nb * R * sizeof(T) + 255) & ~(size_t)255;
    GK_TRY(C->gvecs.ensure(vbytes * (mode == 2 ? 2 : 1)));
    constexpr size_t SLOTS = sizeof(unsigned long long) * GCG_ROUNDS * GCG_VALUES * GCG_MAX_BLOCKS;
    GK_TRY(C->gsync.ensure(SLOTS + 256));
    char* sync = static_cast<char*>(C->gsync.ptr);
    GridCgArgs<V, T> a;
    a.n = n;
    a.R = (int32_t)R;
    a.K = M->K;
    a.stride = M->stride;
    a.col = M->col;
    a.val = (const V*)M->val;
    a.b = b;
    a.x0 = x;
    a.x = mode == 2 ? (T*)(static_cast<char*>(C->gvecs.ptr) + vbytes) : x;
    a.dinv = prec ? (const T*)M->dinv : nullptr;
    a.p = (T*)C->gvecs.ptr;
    a.slots = (unsigned long long*)sync;
    a.arrived = (unsigned long long*)(sync + SLOTS);
    a.err = (int32_t*)(sync + SLOTS + 128);
    a.out = (GridCgOut*)(sync + SLOTS + 192);
    a.tol = tol;
    a.max_iters = max_iters;
    a.inner = inner ? 1 : 0;
    a.stall = inner ? 200 : 0;
    // the hand-offs between blocks take microseconds; a budget below the
    // default must not fail a solve that waits for nothing else
    a.wait_ns = std::max<uint64_t>(M->wait_ns, WAIT_LIMIT_NS);
    const size_t smem = grid_cg_smem<V, T>(mode, R, M->K);
    auto launch = [&](auto kern) -> gk_status {
        GK_TRY(allow_max_dynamic_smem(kern));
        int occ = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, GCG_NT, smem) != cudaSuccess ||
            (int64_t)occ * num_sms() < nb) {
            cudaGetLastError();
            return GK_ERR_UNSUPPORTED;
        }
        GK_CUDA(cudaMemsetAsync(sync, 0xff, SLOTS, s));
        GK_CUDA(cudaMemsetAsync(sync + SLOTS, 0, 256, s));
        void* args[] = {&a};
        const cudaError_t e = cudaLaunchCooperativeKernel((const void*)kern, dim3(nb), dim3(GCG_NT),
                                                          args, smem, s);
        if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
            cudaGetLastError();
            return GK_ERR_UNSUPPORTED;
        }
        GK_CUDA(e);
        return GK_OK;
    };
    auto go = [&](auto md) -> gk_status {
        constexpr int MD = decltype(md)::value;
        return prec ? launch(k_grid_cg<V, T, MD, true>) : launch(k_grid_cg<V, T, MD, false>);
    };
    GridCgOut* h = reinterpret_cast<GridCgOut*>(C->hst);
    static_assert(sizeof(GridCgOut) <= HDR, "the pinned header holds the outcome");
    GK_CUDA(cudaStreamSynchronize(s));
    {
        std::lock_guard<std::mutex> lk(grid_cg_mutex());
        GK_TRY(mode == 0   ? go(std::integral_constant<int, 0>{})
               : mode == 1 ? go(std::integral_constant<int, 1>{})
                           : go(std::integral_constant<int, 2>{}));
        GK_CUDA(cudaMemcpyAsync(h, a.out, sizeof(GridCgOut), cudaMemcpyDeviceToHost, s));
        if (mode == 2)
            GK_CUDA(cudaMemcpyAsync(x, a.x, sizeof(T) * (size_t)n, cudaMemcpyDeviceToDevice, s));
        GK_CUDA(cudaStreamSynchronize(s));
    }
    out->status = (gk_status)h->status;
    out->iters = h->iters;
    out->restarts = h->restarts;
    out->rec = h->rec;
    out->tru = h->tru;
    return GK_OK;
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
