// batched.cu - single-block engine: one thread block runs a whole CG or
// BiCGSTAB solve (same algorithm, stopping rule and residual replacement
// as the multi-kernel engine; Section 3.5 Listings 1-2 for the interface).
//
// Used for many small independent systems in one launch (gk_solve_batched)
// and for small single systems (engine 2).  The vector that SpMV gathers
// from (p for CG; phat, then shat for BiCGSTAB) is staged in shared memory;
// the other vectors live in a per-system global workspace that stays in
// L1/L2.  Blocks loop over systems (persistent grid), so the launch is one
// kernel regardless of the number of systems.  Reductions are block-wide,
// fixed order, so a system's result does not depend on the rest of the
// batch or on the grid size.
#include <cstring>
#include <map>
#include <vector>

#include "prims.cuh"

namespace gk {


// SpMV layouts of a system in the batched engine.  Every layout sums a row
// in its CSR order (one fused multiply-add per stored entry, from zero), so
// the layout never changes a result, only the memory access pattern.
enum BatchLayout : int32_t { BL_CSR = 0, BL_ELL = 1, BL_SELLP = 2 };

struct SysDesc {
    int32_t n, fmt;  // fmt: a BatchLayout
    const int32_t* rp;
    const int32_t* ci;
    const void* va;
    const void* b;
    void* x;
    void* work;  // workspace vectors, each `ld` elements
    int64_t ld;
    double tol;  // this system's relative tolerance
    // padded copy (ELL: K columns of pstride rows; SELL-P: slices of S rows
    // with lengths slen[] and offsets sset[] in units of S entries)
    int32_t* pcol;
    void* pval;
    int32_t* slen;
    int32_t* sset;
    int64_t pstride;
    int32_t K, S;
    int32_t id;  // its place in the caller's arrays
};

// The next system of the batch for this block, -1: none left.  The systems
// are ordered by work, the largest first, and the blocks of the one wave take
// them as they come free: the last ones to run are small.  (Dealt out by
// block index, 2048 systems of 64 to 4096 rows took 20.3 ms and 700 of them
// kept the SMs busy 32 % of the time.)
__device__ __forceinline__ int32_t next_system(int32_t* next, int32_t count) {
    __shared__ int32_t s_next;
    __syncthreads();  // the block is done with the previous system
    if (threadIdx.x == 0) s_next = atomicAdd(next, 1);
    __syncthreads();
    return s_next < count ? s_next : -1;
}

struct SysOut {
    int32_t status, iters, restarts, pad;
    double rec, tru;
};

struct BlockOpts {
    double tol;
    int32_t max_iters;
    int32_t prec;
};

// Reductions use VL virtual lanes: row i adds into lane i mod VL, and the
// VL lane partials are summed by warp 0 in a fixed order.  The rounding of
// every dot product is therefore the same for 128, 256 or 512 threads per
// block, so the block size (autotuned) never changes a system's result.
constexpr int VL = 512;

// per-thread partial sums: NS = VL / threads virtual lanes of NA sums
template <int NA, int NS>
struct VAcc {
    double v[NA][NS] = {};
};

// f(i, s) for every row i of this thread; s = (i mod VL) / NT
template <int NT, class F>
__device__ __forceinline__ void for_rows_vl(int32_t n, F&& f) {
    for (int32_t i0 = threadIdx.x; i0 < n; i0 += VL) {
#pragma unroll
        for (int s = 0; s < VL / NT; ++s) {
            const int32_t i = i0 + s * NT;
            if (i < n) f(i, s);
        }
    }
}

// The reductions' shared memory, one for all of a kernel's sums.
struct SumScratch {
    double sh[2][VL];
    double tot[2];
    int code;
};
__device__ __forceinline__ SumScratch& sum_scratch() {
    __shared__ SumScratch z;
    return z;
}

// Sums the virtual-lane partials over the block; thread 0 runs fin(totals),
// which leaves what follows from them in shared memory, and every thread gets
// its code.  Only thread 0: an FP64 instruction costs the SM 16 cycles per
// warp that issues it, and the divisions and square roots of an iteration
// done by all 16 warps took as long as the rows of a 2,000-row system.
template <int NT, int NA, class Fin>
__device__ __forceinline__ int vl_sum(const VAcc<NA, VL / NT>& acc, Fin&& fin) {
    static_assert(NA <= 2, "the scratch holds two values");
    SumScratch& z = sum_scratch();
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int s = 0; s < VL / NT; ++s) z.sh[a][threadIdx.x + s * NT] = acc.v[a][s];
    __syncthreads();
    // warp a sums value a (each on its own sub-partition's FP64 pipe), lane
    // l lanes l, l + 32, ... as a pairwise tree
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < NA) {
        double t[VL / 32];
#pragma unroll
        for (int k = 0; k < VL / 32; ++k) t[k] = z.sh[warp][lane + 32 * k];
#pragma unroll
        for (int w = VL / 64; w > 0; w >>= 1)
#pragma unroll
            for (int k = 0; k < w; ++k) t[k] += t[k + w];
        const double tt = warp_sum(t[0]);
        if (lane == 0) z.tot[warp] = tt;
    }
    __syncthreads();
    if (threadIdx.x == 0) z.code = fin(z.tot);
    __syncthreads();
    return z.code;
}

// sqrt(t) <= thr (thr >= 0); the square root, ~1,300 cycles, is taken only
// where thr^2 does not already decide
__device__ __forceinline__ bool root_passes(double t, double thr, double thr2) {
    return t <= 1.000001 * thr2 && sqrt(t) <= thr;
}

// What thread 0 keeps of a running solve.
struct BlockScalars {
    double bn, thr, thr2;
    double rho, rho_new, alpha, omega, beta;
    double rec2;  // last squared recurrence residual
    double tru;
};

// A row's len entries at positions p, p + step, ... times the gathered
// vector: four at a time, their columns and values loaded before the gathers
// and those before the first FMA, so a row is one chain of dependent loads
// per four entries.  The one to three left over branch: an FMA that every
// lane skips must not reach the FP64 pipe.  PAD: entries with column -1 (after
// the row's last one) have value 0 and add nothing.
template <bool PAD, typename V, typename T, typename G>
__device__ __forceinline__ T row_chunks(const int32_t* __restrict__ col, const V* __restrict__ val,
                                        const G* __restrict__ g, int64_t p, int64_t step,
                                        int32_t len) {
    T s = T(0);
    auto gather = [&](int32_t c) -> T { return PAD && c < 0 ? T(0) : (T)g[c]; };
    for (; len >= 4; len -= 4, p += 4 * step) {
        int32_t c[4];
        T v[4], x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            c[u] = col[p + u * step];
            v[u] = cvt<T>(val[p + u * step]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = gather(c[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) s = fmadd(v[u], x[u], s);
    }
    if (len > 0) {
        const int32_t c0 = col[p], c1 = len > 1 ? col[p + step] : c0,
                      c2 = len > 2 ? col[p + 2 * step] : c0;
        const T v0 = cvt<T>(val[p]), v1 = len > 1 ? cvt<T>(val[p + step]) : T(0),
                v2 = len > 2 ? cvt<T>(val[p + 2 * step]) : T(0);
        const T x0 = gather(c0);
        if (len > 1) {
            const T x1 = gather(c1);
            if (len > 2) {
                const T x2 = gather(c2);
                s = fmadd(v2, x2, fmadd(v1, x1, fmadd(v0, x0, s)));
            } else {
                s = fmadd(v1, x1, fmadd(v0, x0, s));
            }
        } else {
            s = fmadd(v0, x0, s);
        }
    }
    return s;
}

// Row i of a system in its layout (see BatchLayout): entries in CSR order,
// padding (column -1) only after a row's last entry.
// L = BL_CSR: every system of the batch (the branch is resolved at compile
// time); L = -1: the layout is read per system.
template <typename V, typename T, int L, typename G>
__device__ __forceinline__ T sys_row_dot(const SysDesc& d, const G* __restrict__ g, int32_t i) {
    const int fmt = L >= 0 ? L : d.fmt;
    if (fmt == BL_ELL)
        return row_chunks<true, V, T>(d.pcol, (const V*)d.pval, g, i, d.pstride, d.K);
    if (fmt == BL_SELLP) {
        const int32_t sl = i / d.S, t = i - sl * d.S;
        return row_chunks<true, V, T>(d.pcol, (const V*)d.pval, g, (int64_t)d.sset[sl] * d.S + t,
                                      (int64_t)d.S, d.slen[sl]);
    }
    const int32_t a = d.rp[i];
    return row_chunks<false, V, T>(d.ci, (const V*)d.va, g, a, 1, d.rp[i + 1] - a);
}

// Writes the padded copy of every system whose layout is ELL or SELL-P
// (one block per system, grid-stride over systems).  SELL-P: slice lengths
// (longest row of the slice), then their exclusive scan, then the entries.
template <typename V>
__global__ void __launch_bounds__(256) k_batch_pad(SysDesc* __restrict__ sys, int32_t count) {
    for (int32_t sidx = blockIdx.x; sidx < count; sidx += gridDim.x) {
        SysDesc& d = sys[sidx];
        if (d.fmt == BL_CSR) continue;
        const int32_t n = d.n;
        const V* __restrict__ va = (const V*)d.va;
        V* __restrict__ pv = (V*)d.pval;
        if (d.fmt == BL_ELL) {
            for (int64_t i = threadIdx.x; i < d.pstride; i += blockDim.x) {
                const int32_t a = i < n ? d.rp[i] : 0, e = i < n ? d.rp[i + 1] : 0;
                for (int32_t k = 0; k < d.K; ++k) {
                    const int64_t p = (int64_t)k * d.pstride + i;
                    const bool in = a + k < e;
                    d.pcol[p] = in ? d.ci[a + k] : -1;
                    pv[p] = in ? va[a + k] : V(0.0f);
                }
            }
            continue;
        }
        const int32_t S = d.S, ns = (n + S - 1) / S;
        for (int32_t sl = threadIdx.x; sl < ns; sl += blockDim.x) {
            int32_t mx = 0;
            for (int32_t t = 0; t < S; ++t) {
                const int32_t i = sl * S + t;
                if (i < n) mx = max(mx, d.rp[i + 1] - d.rp[i]);
            }
            d.slen[sl] = mx;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int32_t acc = 0;
            for (int32_t sl = 0; sl < ns; ++sl) {
                d.sset[sl] = acc;
                acc += d.slen[sl];
            }
            d.sset[ns] = acc;
        }
        __syncthreads();
        for (int64_t i = threadIdx.x; i < (int64_t)ns * S; i += blockDim.x) {
            const int32_t sl = (int32_t)(i / S), t = (int32_t)(i - (int64_t)sl * S);
            const int32_t a = i < n ? d.rp[i] : 0, e = i < n ? d.rp[i + 1] : 0;
            const int64_t base = (int64_t)d.sset[sl] * S + t;
            for (int32_t k = 0; k < d.slen[sl]; ++k) {
                const int64_t p = base + (int64_t)k * S;
                const bool in = a + k < e;
                d.pcol[p] = in ? d.ci[a + k] : -1;
                pv[p] = in ? va[a + k] : V(0.0f);
            }
        }
        __syncthreads();
    }
}

// Jacobi inverse diagonal of row i; 0 when missing or zero.
template <typename V, typename T>
__device__ __forceinline__ T row_dinv(const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                      const V* __restrict__ va, int32_t i) {
    T d = T(0);
    for (int32_t k = rp[i]; k < rp[i + 1]; ++k)
        if (ci[k] == i) d += cvt<T>(va[k]);
    return d == T(0) ? T(0) : T(1) / d;
}

// why a block's solve ends (0: it goes on)
enum : int { BE_OK = 1, BE_PASSED, BE_NAN, BE_BREAKDOWN, BE_ZERO_DIAG, BE_ZERO_RHS };

// r = b - A x in place; BE_OK when ||r|| <= thr, BE_NAN when not finite
template <typename V, typename T, int L, int NT>
__device__ int block_true_resid(const SysDesc& d, T* r, BlockScalars& S) {
    const T* b = (const T*)d.b;
    const T* x = (const T*)d.x;
    VAcc<1, VL / NT> tt;
    for_rows_vl<NT>(d.n, [&](int32_t i, int s) {
        const T ri = b[i] - sys_row_dot<V, T, L>(d, x, i);
        r[i] = ri;
        tt.v[0][s] = fma((double)ri, (double)ri, tt.v[0][s]);
    });
    return vl_sum<NT>(tt, [&](const double* t) -> int {
        const double tn = sqrt(t[0]);
        S.tru = tn / S.bn;
        return !isfinite(tn) ? BE_NAN : tn <= S.thr ? BE_OK : 0;
    });
}

// Prepares a system: Jacobi diagonal (in work slot 0), ||b||, true residual.
template <typename V, typename T, int L, int NT>
__device__ int block_setup(const SysDesc& d, const BlockOpts& opt, T* dinv, T* r,
                           BlockScalars& S) {
    const int32_t n = d.n;
    const V* va = (const V*)d.va;
    const T* b = (const T*)d.b;
    T* x = (T*)d.x;
    VAcc<2, VL / NT> acc;
    for_rows_vl<NT>(n, [&](int32_t i, int s) {
        const T bi = b[i];
        acc.v[0][s] = fma((double)bi, (double)bi, acc.v[0][s]);
        if (opt.prec) {
            const T di = row_dinv<V, T>(d.rp, d.ci, va, i);
            dinv[i] = di;
            if (di == T(0)) acc.v[1][s] = 1.0;
        }
    });
    const int code = vl_sum<NT>(acc, [&](const double* t) -> int {
        S.tru = S.rec2 = 0.0;
        S.bn = sqrt(t[0]);
        S.thr = d.tol * S.bn;
        S.thr2 = S.thr * S.thr;
        return t[1] != 0.0 ? BE_ZERO_DIAG : S.bn == 0.0 ? BE_ZERO_RHS : !isfinite(S.bn) ? BE_NAN : 0;
    });
    if (code == BE_ZERO_RHS)
        for (int32_t i = threadIdx.x; i < n; i += NT) x[i] = T(0);
    if (code != 0) return code;
    const int res = block_true_resid<V, T, L, NT>(d, r, S);
    if (threadIdx.x == 0) S.rec2 = -1.0;  // no recurrence yet: its residual is the true one
    return res;
}

// The outcome of a solve that ended with `end` (0: at the iteration cap).
__device__ __forceinline__ SysOut block_outcome(int end, int32_t iters, int32_t restarts,
                                                double first_true, const BlockScalars& S) {
    SysOut o;
    o.status = end == BE_OK || end == BE_ZERO_RHS ? GK_OK
               : end == BE_NAN                    ? GK_ERR_NAN
               : end == BE_BREAKDOWN              ? GK_BREAKDOWN
               : end == BE_ZERO_DIAG              ? GK_ERR_ZERO_DIAG
                                                  : GK_NOT_CONVERGED;
    o.iters = iters;
    o.restarts = restarts;
    o.pad = 0;
    o.tru = S.tru;
    o.rec = S.rec2 < 0.0 ? first_true : S.rec2 > 0.0 || S.rec2 != S.rec2 ? sqrt(S.rec2) / S.bn : 0.0;
    return o;
}

// ---------------------------------------------------------------- CG
// work slots: 0 dinv, 1 r, 2 q, 3 scratch (final residual)
constexpr int BLOCK_MAX_THREADS = 512;

template <typename V, typename T, int L, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_block_cg(const SysDesc* __restrict__ sys, SysOut* __restrict__ outs,
                           int32_t count, int32_t* next, BlockOpts opt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ BlockScalars S;
    T* ps = reinterpret_cast<T*>(smem_raw);
    for (int32_t sidx; (sidx = next_system(next, count)) >= 0;) {
        const SysDesc d = sys[sidx];
        const int32_t n = d.n;
        T* x = (T*)d.x;
        T* dinv = (T*)d.work;
        T* r = dinv + d.ld;
        T* q = r + d.ld;
        T* scratch = q + d.ld;
        int32_t k = 0, restarts = 0;
        int end = block_setup<V, T, L, NT>(d, opt, dinv, r, S);
        const double first_true = S.tru;
        const bool run = end == 0;
        auto init_dir = [&]() {
            VAcc<1, VL / NT> rz;
            for_rows_vl<NT>(n, [&](int32_t i, int s) {
                const T ri = r[i];
                const T zi = opt.prec ? dinv[i] * ri : ri;
                ps[i] = zi;
                rz.v[0][s] = fma((double)ri, (double)zi, rz.v[0][s]);
            });
            vl_sum<NT>(rz, [&](const double* t) {
                S.rho = t[0];
                return 0;
            });
        };
        if (run) init_dir();
        while (end == 0 && k < opt.max_iters) {
            VAcc<1, VL / NT> pq;
            for_rows_vl<NT>(n, [&](int32_t i, int s) {
                const T sv = sys_row_dot<V, T, L>(d, ps, i);
                q[i] = sv;
                pq.v[0][s] = fma((double)ps[i], (double)sv, pq.v[0][s]);
            });
            end = vl_sum<NT>(pq, [&](const double* t) -> int {
                S.alpha = S.rho / t[0];
                return !isfinite(t[0]) ? BE_NAN : t[0] <= 0.0 ? BE_BREAKDOWN : 0;
            });
            if (end != 0) break;
            const T ta = (T)S.alpha;
            VAcc<2, VL / NT> a2;
            for_rows_vl<NT>(n, [&](int32_t i, int s) {
                x[i] = fmadd(ta, ps[i], x[i]);
                const T ri = fmadd(-ta, q[i], r[i]);
                r[i] = ri;
                const T zi = opt.prec ? dinv[i] * ri : ri;
                if (opt.prec) q[i] = zi;  // q has been used: z waits there for beta
                a2.v[0][s] = fma((double)ri, (double)zi, a2.v[0][s]);
                a2.v[1][s] = fma((double)ri, (double)ri, a2.v[1][s]);
            });
            end = vl_sum<NT>(a2, [&](const double* t) -> int {
                S.rec2 = t[1];
                if (!isfinite(t[1]) || !isfinite(t[0])) return BE_NAN;
                if (root_passes(t[1], S.thr, S.thr2)) return BE_PASSED;
                S.beta = t[0] / S.rho;
                S.rho = t[0];
                return 0;
            });
            ++k;
            if (end == BE_PASSED) {
                // the true residual decides; a NaN there ends no solve here
                end = block_true_resid<V, T, L, NT>(d, r, S) == BE_OK ? BE_OK : 0;
                if (end != 0) break;
                restarts += 1;  // residual replacement, restart from x
                init_dir();
                continue;
            }
            if (end != 0) break;
            const T tb = (T)S.beta;
            for (int32_t i = threadIdx.x; i < n; i += NT)
                ps[i] = fmadd(tb, ps[i], opt.prec ? q[i] : r[i]);
            __syncthreads();
        }
        if (run) block_true_resid<V, T, L, NT>(d, scratch, S);
        if (threadIdx.x == 0) outs[d.id] = block_outcome(end, k, restarts, first_true, S);
    }
}

// ---------------------------------------------------------------- BiCGSTAB
// work slots: 0 dinv, 1 r, 2 rhat, 3 p, 4 phat, 5 v, 6 s, 7 shat, 8 t
template <typename V, typename T, int L, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_block_bicgstab(const SysDesc* __restrict__ sys, SysOut* __restrict__ outs,
                                 int32_t count, int32_t* next, BlockOpts opt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ BlockScalars S;
    T* gs = reinterpret_cast<T*>(smem_raw);  // gathered vector
    for (int32_t sidx; (sidx = next_system(next, count)) >= 0;) {
        const SysDesc d = sys[sidx];
        const int32_t n = d.n;
        T* x = (T*)d.x;
        T* dinv = (T*)d.work;
        T *r = dinv + d.ld, *rh = r + d.ld, *p = rh + d.ld, *ph = p + d.ld, *v = ph + d.ld;
        T *sv = v + d.ld, *sh = sv + d.ld, *t = sh + d.ld;
        int32_t k = 0, restarts = 0;
        int end = block_setup<V, T, L, NT>(d, opt, dinv, r, S);
        const double first_true = S.tru;
        const bool run = end == 0;
        // beta of the next step from rho', or why there is none
        auto next_beta = [&]() -> int {
            if (!isfinite(S.rho_new)) return BE_NAN;
            if (S.rho_new == 0.0) return BE_BREAKDOWN;
            S.beta = (S.rho_new / S.rho) * (S.alpha / S.omega);
            return 0;
        };
        auto restart = [&]() -> int {
            VAcc<1, VL / NT> a;
            for_rows_vl<NT>(n, [&](int32_t i, int s) {
                const T ri = r[i];
                rh[i] = ri;
                p[i] = T(0);
                v[i] = T(0);
                a.v[0][s] = fma((double)ri, (double)ri, a.v[0][s]);
            });
            return vl_sum<NT>(a, [&](const double* tt) -> int {
                S.rho = S.alpha = S.omega = 1.0;
                S.rho_new = tt[0];
                return next_beta();
            });
        };
        // the true residual decides a passed recurrence residual: 0 and a
        // restart from it when it fails
        auto confirm = [&]() -> int {
            if (block_true_resid<V, T, L, NT>(d, r, S) == BE_OK) return BE_OK;
            restarts += 1;
            return restart();
        };
        if (run) end = restart();
        // what stops a step (NaN, breakdown) counts only while steps are left
        if (run && opt.max_iters <= 0) end = 0;
        while (end == 0 && k < opt.max_iters) {
            {
                const T beta = (T)S.beta, tw = (T)S.omega;
                for (int32_t i = threadIdx.x; i < n; i += NT) {
                    const T pi = fmadd(beta, fmadd(-tw, v[i], p[i]), r[i]);
                    p[i] = pi;
                    const T hi = opt.prec ? dinv[i] * pi : pi;
                    ph[i] = hi;
                    gs[i] = hi;
                }
            }
            __syncthreads();
            VAcc<1, VL / NT> rv;
            for_rows_vl<NT>(n, [&](int32_t i, int s) {
                const T vi = sys_row_dot<V, T, L>(d, gs, i);
                v[i] = vi;
                rv.v[0][s] = fma((double)rh[i], (double)vi, rv.v[0][s]);
            });
            end = vl_sum<NT>(rv, [&](const double* tt) -> int {
                S.alpha = S.rho_new / tt[0];
                return !isfinite(tt[0]) ? BE_NAN : tt[0] == 0.0 ? BE_BREAKDOWN : 0;
            });
            if (end != 0) break;
            const T ta = (T)S.alpha;
            VAcc<1, VL / NT> ss;
            for_rows_vl<NT>(n, [&](int32_t i, int s) {
                const T si = fmadd(-ta, v[i], r[i]);
                sv[i] = si;
                ss.v[0][s] = fma((double)si, (double)si, ss.v[0][s]);
            });
            ++k;
            end = vl_sum<NT>(ss, [&](const double* tt) -> int {
                if (!isfinite(tt[0])) return BE_NAN;
                if (!root_passes(tt[0], S.thr, S.thr2)) return 0;
                S.rec2 = tt[0];
                return BE_PASSED;
            });
            if (end == BE_PASSED) {  // half-step exit
                for (int32_t i = threadIdx.x; i < n; i += NT) x[i] = fmadd(ta, ph[i], x[i]);
                __syncthreads();
                end = confirm();
                if (end > 0 && end != BE_OK && k >= opt.max_iters) end = 0;
                continue;
            }
            if (end != 0) break;
            for (int32_t i = threadIdx.x; i < n; i += NT) {
                const T hi = opt.prec ? dinv[i] * sv[i] : sv[i];
                sh[i] = hi;
                gs[i] = hi;
            }
            __syncthreads();
            VAcc<2, VL / NT> a2;
            for_rows_vl<NT>(n, [&](int32_t i, int s) {
                const T ti = sys_row_dot<V, T, L>(d, gs, i);
                t[i] = ti;
                a2.v[0][s] = fma((double)ti, (double)sv[i], a2.v[0][s]);
                a2.v[1][s] = fma((double)ti, (double)ti, a2.v[1][s]);
            });
            end = vl_sum<NT>(a2, [&](const double* tt) -> int {
                if (!isfinite(tt[0]) || !isfinite(tt[1])) return BE_NAN;
                if (tt[1] == 0.0) return BE_BREAKDOWN;
                S.omega = tt[0] / tt[1];
                return S.omega == 0.0 ? BE_BREAKDOWN : 0;
            });
            if (end != 0) break;
            const T to = (T)S.omega;
            VAcc<2, VL / NT> a3;
            for_rows_vl<NT>(n, [&](int32_t i, int s) {
                x[i] = fmadd(to, sh[i], fmadd(ta, ph[i], x[i]));
                const T ri = fmadd(-to, t[i], sv[i]);
                r[i] = ri;
                a3.v[0][s] = fma((double)rh[i], (double)ri, a3.v[0][s]);
                a3.v[1][s] = fma((double)ri, (double)ri, a3.v[1][s]);
            });
            end = vl_sum<NT>(a3, [&](const double* tt) -> int {
                S.rho = S.rho_new;
                S.rho_new = tt[0];
                S.rec2 = tt[1];
                if (!isfinite(tt[1])) return BE_NAN;
                if (root_passes(tt[1], S.thr, S.thr2)) return BE_PASSED;
                return k < opt.max_iters ? next_beta() : 0;
            });
            if (end == BE_PASSED) {
                end = confirm();
                if (end > 0 && end != BE_OK && k >= opt.max_iters) end = 0;
            }
        }
        if (run) block_true_resid<V, T, L, NT>(d, t, S);
        if (threadIdx.x == 0) outs[d.id] = block_outcome(end, k, restarts, first_true, S);
    }
}

// ---------------------------------------------------------------- host

static int nslots(int method) { return method == GK_CG ? 4 : 9; }

// Layout policy of a batch (picked by the autotuner per batch shape):
// layout BL_CSR runs every system on its CSR arrays; BL_ELL gives each system
// an ELL copy when ELL stores at most 1.2 x its nonzeros, else keeps its
// CSR; BL_SELLP gives each system a SELL-P copy with slices of S rows.
// nt: threads per block.  The untuned default (batches of fewer than
// TUNE_MIN_COUNT systems) is CSR: on lone serving-size systems (n 1,575 to
// 13,689; stencils and banded SPD) it took 0.31-0.65x the time of ELL or
// SELL-P(32) in the one-block kernel.
constexpr int32_t TUNE_MIN_COUNT = 64;  // smallest batch the autotuner times

// Threads per block where the largest system decides: 512 above this many
// rows, below it 256, or what the autotuner times of the two.  A batch ends
// with its slowest systems alone on their SMs, where twice the threads hide
// twice the latency; the tuner's short trials do not see that end.  ms with
// 256 / 512 threads, FP64: 2048 systems of up to 4096 rows 10.1 / 7.1, 700
// 6.2 / 4.0, 20 2.7 / 1.9, one of 1881 rows 1.5 / 1.0; 1500 of up to 1024
// rows 1.7 / 1.8; FP32: 4.2 / 2.9, 2.6 / 1.7, 1.1 / 0.75, 0.42 / 0.37; 0.77 /
// 0.82.  (128 threads: 1.4 to 2.4 times as long as 256.)
constexpr int32_t WIDE_BLOCK_ROWS = 1024;

struct BatchCfg {
    int nt = 256;
    int layout = BL_CSR;
    int S = 32;
};

struct BatchBufs {
    DevBuf desc, outs, work, pad;
    SysDesc* hdesc = nullptr;
    SysOut* hout = nullptr;      // hcap outcomes, then hcap indices: the order of the systems
    size_t hcap = 0;
    ~BatchBufs() {
        if (hdesc) cudaFreeHost(hdesc);
        if (hout) cudaFreeHost(hout);
        desc.release();
        outs.release();
        work.release();
        pad.release();
    }
};

// Buffers are pooled: a call takes a free set (or makes one) and returns it,
// so batches launched from different host threads run concurrently.
static std::mutex g_batch_mu;
static std::vector<BatchBufs*> g_batch_pool;

struct BatchLease {
    BatchBufs* b = nullptr;
    BatchLease() {
        std::lock_guard<std::mutex> lk(g_batch_mu);
        if (!g_batch_pool.empty()) {
            b = g_batch_pool.back();
            g_batch_pool.pop_back();
        }
        if (!b) b = new BatchBufs();
    }
    ~BatchLease() {
        std::lock_guard<std::mutex> lk(g_batch_mu);
        g_batch_pool.push_back(b);
    }
};

// The block kernel for a method, value type, batch layout (every system
// CSR, or -1: read per system) and block size.
template <typename V, typename T, int L, int NT>
static auto block_kernel(int method) {
    return method == GK_CG ? k_block_cg<V, T, L, NT> : k_block_bicgstab<V, T, L, NT>;
}

template <typename V, typename T>
static auto block_kernel(int method, int lay, int nt) {
    if (lay == BL_CSR)
        return nt == 128   ? block_kernel<V, T, BL_CSR, 128>(method)
               : nt == 256 ? block_kernel<V, T, BL_CSR, 256>(method)
                           : block_kernel<V, T, BL_CSR, 512>(method);
    return nt == 128   ? block_kernel<V, T, -1, 128>(method)
           : nt == 256 ? block_kernel<V, T, -1, 256>(method)
                       : block_kernel<V, T, -1, 512>(method);
}

template <typename V, typename T>
static gk_status launch_block(int method, int lay, const SysDesc* ddesc, SysOut* dout,
                              int32_t count, int32_t* next, const BlockOpts& bo, int nt,
                              size_t smem, unsigned grid, cudaStream_t s) {
    auto k = block_kernel<V, T>(method, lay, nt);
    GK_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    k<<<grid, nt, smem, s>>>(ddesc, dout, count, next, bo);
    GK_CUDA(cudaGetLastError());
    return GK_OK;
}

static size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

// Layout of system A under a policy, and the bytes of its padded copy.
static int sys_layout(const gk_matrix A, const BatchCfg& cfg, size_t* pad_bytes) {
    *pad_bytes = 0;
    if (A->n == 0 || A->nnz == 0 || cfg.layout == BL_CSR) return BL_CSR;
    const size_t sv = value_bytes(A->dtype);
    if (cfg.layout == BL_ELL) {
        const int64_t stride = ((int64_t)A->n + 31) / 32 * 32;
        if ((int64_t)A->max_row * A->n > A->nnz + A->nnz / 5) return BL_CSR;
        *pad_bytes = al256((size_t)A->max_row * stride * 4) + al256((size_t)A->max_row * stride * sv);
        return BL_ELL;
    }
    // SELL-P: at most the longest row in every slice
    const int64_t ns = ((int64_t)A->n + cfg.S - 1) / cfg.S;
    const size_t ent = (size_t)ns * cfg.S * A->max_row;
    *pad_bytes = al256(ent * 4) + al256(ent * sv) + al256(4 * (size_t)ns) + al256(4 * (size_t)(ns + 1));
    return BL_SELLP;
}

// Runs count systems; infos may be null.  All matrices CSR, same dtype.
static gk_status run_batch(int32_t count, const gk_matrix* As, const void* const* bs,
                           void* const* xs, const gk_solve_opts* o, gk_solve_info* infos,
                           cudaStream_t s, const BatchCfg& cfg, float* ms_out) {
    const int nt = cfg.nt;
    const gk_dtype dt = As[0]->dtype;
    const size_t vb = vector_bytes(dt);
    int32_t nmax = 0;
    size_t wbytes = 0, pbytes = 0;
    const int ns = nslots(o->method);
    for (int32_t i = 0; i < count; ++i) {
        nmax = std::max(nmax, As[i]->n);
        const size_t ld = (((size_t)As[i]->n * vb + 255) & ~(size_t)255) / vb;
        wbytes += ld * vb * ns;
        size_t pb = 0;
        sys_layout(As[i], cfg, &pb);
        pbytes += pb;
    }
    const size_t smem = std::max<size_t>((size_t)nmax * vb, 16);
    if (smem > 200 * 1024) return GK_ERR_UNSUPPORTED;
    BatchLease lease;
    BatchBufs& B = *lease.b;
    if (B.hcap < (size_t)count) {
        GateShared gate;
        if (B.hdesc) cudaFreeHost(B.hdesc);
        if (B.hout) cudaFreeHost(B.hout);
        B.hdesc = nullptr;
        B.hout = nullptr;
        B.hcap = 0;
        GK_CUDA(cudaMallocHost(&B.hdesc, sizeof(SysDesc) * (size_t)count));
        GK_CUDA(cudaMallocHost(&B.hout, (sizeof(SysOut) + sizeof(int32_t)) * (size_t)count));
        B.hcap = (size_t)count;
    }
    GK_TRY(B.desc.ensure(sizeof(SysDesc) * (size_t)count));
    GK_TRY(B.outs.ensure(sizeof(SysOut) * (size_t)count + 16));
    GK_TRY(B.work.ensure(wbytes + 256));
    if (pbytes) GK_TRY(B.pad.ensure(pbytes + 256));
    char* w = (char*)B.work.ptr;
    char* pw = (char*)B.pad.ptr;
    bool any_pad = false;
    int32_t* order = (int32_t*)(B.hout + B.hcap);  // the largest system first
    for (int32_t i = 0; i < count; ++i) order[i] = i;
    auto work = [&](int32_t i) { return As[i]->nnz + 8 * (int64_t)As[i]->n; };
    std::sort(order, order + count, [&](int32_t a, int32_t b) {
        return work(a) != work(b) ? work(a) > work(b) : a < b;
    });
    for (int32_t k = 0; k < count; ++k) {
        const int32_t i = order[k];
        gk_matrix A = As[i];
        SysDesc& d = B.hdesc[k];
        std::memset(&d, 0, sizeof(d));
        d.id = i;
        d.n = A->n;
        size_t pb = 0;
        d.fmt = sys_layout(A, cfg, &pb);
        if (d.fmt == BL_ELL) {
            d.K = A->max_row;
            d.pstride = ((int64_t)A->n + 31) / 32 * 32;
            d.pcol = (int32_t*)pw;
            d.pval = pw + al256((size_t)d.K * d.pstride * 4);
        } else if (d.fmt == BL_SELLP) {
            d.S = cfg.S;
            d.K = A->max_row;
            const int64_t nsl = ((int64_t)A->n + cfg.S - 1) / cfg.S;
            const size_t ent = (size_t)nsl * cfg.S * A->max_row;
            d.pcol = (int32_t*)pw;
            d.pval = pw + al256(ent * 4);
            d.slen = (int32_t*)(pw + al256(ent * 4) + al256(ent * value_bytes(A->dtype)));
            d.sset = d.slen + al256(4 * (size_t)nsl) / 4;
        }
        pw += pb;
        any_pad |= d.fmt != BL_CSR;
        d.rp = A->row_ptr;
        d.ci = A->col;
        d.va = A->val;
        d.b = bs[i];
        d.x = xs[i];
        d.work = w;
        d.ld = (int64_t)((((size_t)A->n * vb + 255) & ~(size_t)255) / vb);
        d.tol = o->batch_tols ? o->batch_tols[i] : o->tol;
        w += (size_t)d.ld * vb * ns;
    }
    int32_t* next = (int32_t*)((SysOut*)B.outs.ptr + count);
    GK_CUDA(cudaMemsetAsync(next, 0, sizeof(int32_t), s));
    GK_CUDA(cudaMemcpyAsync(B.desc.ptr, B.hdesc, sizeof(SysDesc) * (size_t)count,
                            cudaMemcpyHostToDevice, s));
    BlockOpts bo{o->tol, o->max_iters, o->precond == GK_PRECOND_JACOBI};
    int occ = 1;
    const int sms = num_sms();
    cudaEvent_t e0, e1;
    GK_CUDA(cudaEventCreate(&e0));
    GK_CUDA(cudaEventCreate(&e1));
    GK_CUDA(cudaEventRecord(e0, s));
    gk_status st = GK_OK;
    if (any_pad) {  // the padded copies of this batch, one block per system
        const unsigned pg = (unsigned)std::min<int64_t>(count, (int64_t)sms * 8);
        SysDesc* dd = (SysDesc*)B.desc.ptr;
        if (dt == GK_F64) k_batch_pad<double><<<pg, 256, 0, s>>>(dd, count);
        else if (dt == GK_F32) k_batch_pad<float><<<pg, 256, 0, s>>>(dd, count);
        else k_batch_pad<__nv_bfloat16><<<pg, 256, 0, s>>>(dd, count);
        GK_CUDA(cudaGetLastError());
    }
    auto occ_of = [&](auto kern) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        int b = 1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, nt, smem) != cudaSuccess || b < 1) b = 1;
        return b;
    };
    // one layout for the whole batch: the kernel without the per-row branch
    int lay = count > 0 ? B.hdesc[0].fmt : BL_CSR;
    for (int32_t i = 1; i < count && lay >= 0; ++i)
        if (B.hdesc[i].fmt != lay) lay = -1;
    if (dt == GK_F64) occ = occ_of(block_kernel<double, double>(o->method, lay, nt));
    else if (dt == GK_F32) occ = occ_of(block_kernel<float, float>(o->method, lay, nt));
    else occ = occ_of(block_kernel<__nv_bfloat16, float>(o->method, lay, nt));
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(count, (int64_t)sms * occ));
    const SysDesc* dd = (const SysDesc*)B.desc.ptr;
    SysOut* dout = (SysOut*)B.outs.ptr;
    if (dt == GK_F64)
        st = launch_block<double, double>(o->method, lay, dd, dout, count, next, bo, nt, smem, grid, s);
    else if (dt == GK_F32)
        st = launch_block<float, float>(o->method, lay, dd, dout, count, next, bo, nt, smem, grid, s);
    else
        st = launch_block<__nv_bfloat16, float>(o->method, lay, dd, dout, count, next, bo, nt,
                                                smem, grid, s);
    GK_CUDA(cudaEventRecord(e1, s));
    if (st == GK_OK) {
        GK_CUDA(cudaMemcpyAsync(B.hout, B.outs.ptr, sizeof(SysOut) * (size_t)count,
                                cudaMemcpyDeviceToHost, s));
        GK_CUDA(cudaStreamSynchronize(s));
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms_out) *ms_out = ms;
        if (infos)
            for (int32_t k = 0; k < count; ++k) {
                const int32_t i = B.hdesc[k].id;
                const SysOut& so = B.hout[i];
                infos[i].status = (gk_status)so.status;
                infos[i].iters = so.iters;
                infos[i].restarts = so.restarts;
                infos[i].outer_iters = 0;
                infos[i].rel_res_recurrence = so.rec;
                infos[i].rel_res_true = so.tru;
                infos[i].device_ms = ms;
                infos[i].spmv_format = B.hdesc[k].fmt == BL_ELL     ? GK_ELL
                                       : B.hdesc[k].fmt == BL_SELLP ? GK_SELLP
                                                                    : GK_CSR;
                infos[i].block_threads = nt;
                infos[i].slice_size = B.hdesc[k].fmt == BL_SELLP ? cfg.S : 0;
            }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return st;
}


gk_status solve_small(gk_matrix A, const void* b, void* x, const gk_solve_opts* o, cudaStream_t s,
                      SolveOut* out) {
    if (A->fmt != GK_CSR || o->method == GK_GMRES || o->method == GK_CGS || A->dtype == GK_F16 ||
        o->precond >= GK_PRECOND_BLOCK_JACOBI)
        return GK_ERR_UNSUPPORTED;
    gk_solve_info info;
    std::memset(&info, 0, sizeof(info));
    gk_matrix As[1] = {A};
    const void* bs[1] = {b};
    void* xs[1] = {x};
    BatchCfg cfg;
    cfg.nt = BLOCK_MAX_THREADS;
    GK_TRY(run_batch(1, As, bs, xs, o, &info, s, cfg, nullptr));
    out->status = info.status;
    out->iters = info.iters;
    out->restarts = info.restarts;
    out->rec = info.rel_res_recurrence;
    out->tru = info.rel_res_true;
    out->layout = info.spmv_format;
    out->slice = info.slice_size;
    out->threads = info.block_threads;
    return GK_OK;
}

// ------------------------------------------------------------ autotuner
// The configuration of a batch shape -- each system's SpMV layout (policy
// CSR, ELL where its padding is at most 20 %, or SELL-P with slices of
// S = 8, 16 or 32 rows) and, for small systems (see WIDE_BLOCK_ROWS), the
// threads per block (256 or 512) -- is picked by timing
// every candidate on a run of the batch itself capped at 30 iterations (the
// callers' initial guesses are saved before and restored after the trials)
// and cached per key: value type, method, preconditioner, log2 of the
// largest n and of the system count.  No candidate changes a result: every
// layout sums a row in CSR order and the reductions use fixed virtual lanes.
static std::mutex g_tune_mu;
static std::map<uint64_t, BatchCfg> g_tune;

static uint64_t tune_key(gk_dtype dt, const gk_solve_opts* o, int32_t nmax, int32_t count) {
    auto lg = [](int64_t v) {
        int b = 0;
        while ((1ll << b) < v) ++b;
        return (uint64_t)b;
    };
    return ((uint64_t)dt << 40) | ((uint64_t)o->method << 36) | ((uint64_t)o->precond << 32) |
           (lg(nmax) << 16) | lg(count);
}

static gk_status autotune(int32_t count, const gk_matrix* As, const void* const* bs,
                          void* const* xs, const gk_solve_opts* o, cudaStream_t s,
                          BatchCfg* best) {
    const size_t vb = vector_bytes(As[0]->dtype);
    size_t total = 0;
    for (int32_t i = 0; i < count; ++i) total += (size_t)As[i]->n * vb;
    DevBuf save;
    GK_TRY(save.ensure(total + 256));
    auto copy_all = [&](bool to_save) -> gk_status {
        size_t off = 0;
        for (int32_t i = 0; i < count; ++i) {
            const size_t b = (size_t)As[i]->n * vb;
            char* sp = static_cast<char*>(save.ptr) + off;
            if (b)
                GK_CUDA(cudaMemcpyAsync(to_save ? (void*)sp : xs[i], to_save ? xs[i] : (void*)sp, b,
                                        cudaMemcpyDeviceToDevice, s));
            off += b;
        }
        return GK_OK;
    };
    GK_TRY(copy_all(true));
    gk_solve_opts trial = *o;
    trial.max_iters = std::min(o->max_iters, 30);
    float best_ms = 1e30f;
    *best = BatchCfg();
    const int layouts[5][2] = {{BL_CSR, 0}, {BL_ELL, 0}, {BL_SELLP, 8}, {BL_SELLP, 16}, {BL_SELLP, 32}};
    int32_t nmax = 0;
    for (int32_t i = 0; i < count; ++i) nmax = std::max(nmax, As[i]->n);
    for (const auto& L : layouts)
        for (int nt : {256, 512}) {
            if (nt == 256 && nmax > WIDE_BLOCK_ROWS) continue;
            BatchCfg c;
            c.layout = L[0];
            c.S = L[0] == BL_SELLP ? L[1] : 32;
            c.nt = nt;
            GK_TRY(copy_all(false));
            float ms = 0.f;
            GK_TRY(run_batch(count, As, bs, xs, &trial, nullptr, s, c, &ms));
            if (ms < best_ms) {
                best_ms = ms;
                *best = c;
            }
        }
    GK_TRY(copy_all(false));
    GK_CUDA(cudaStreamSynchronize(s));
    save.release();
    return GK_OK;
}

// GK_BATCH_LAYOUT = csr | ell | sellp8 | sellp16 | sellp32 | sellp64 forces a layout
// policy; GK_BATCH_THREADS = 128 | 256 | 512 forces the block size.
static bool forced_layout(BatchCfg* c) {
    const char* e = getenv("GK_BATCH_LAYOUT");
    if (!e) return false;
    if (!strcmp(e, "csr")) c->layout = BL_CSR;
    else if (!strcmp(e, "ell")) c->layout = BL_ELL;
    else if (!strncmp(e, "sellp", 5)) {
        const int S = atoi(e + 5);
        if (S != 8 && S != 16 && S != 32 && S != 64) return false;
        c->layout = BL_SELLP;
        c->S = S;
    } else {
        return false;
    }
    return true;
}

}  // namespace gk

using namespace gk;

extern "C" gk_status gk_solve_batched(int32_t count, const gk_matrix* As, const void* const* bs,
                                      void* const* xs, const gk_solve_opts* o,
                                      gk_solve_info* infos, void* stream) {
    if (count < 0 || !o || (count > 0 && (!As || !bs || !xs))) return GK_ERR_INVALID;
    if (count == 0) return GK_OK;
    if (o->method == GK_GMRES || o->method == GK_CGS || o->precond >= GK_PRECOND_BLOCK_JACOBI)
        return GK_ERR_UNSUPPORTED;
    if ((o->method != GK_CG && o->method != GK_BICGSTAB) || o->mixed ||
        (o->precond != GK_PRECOND_NONE && o->precond != GK_PRECOND_JACOBI) || !(o->tol >= 0.0) ||
        o->max_iters < 0)
        return GK_ERR_INVALID;
    if (o->batch_tols)
        for (int32_t i = 0; i < count; ++i)
            if (!(o->batch_tols[i] >= 0.0)) return GK_ERR_INVALID;
    int dev = -1;
    cudaGetDevice(&dev);
    for (int32_t i = 0; i < count; ++i) {
        const gk_matrix A = As[i];
        if (A && A->dtype == GK_F16) return GK_ERR_UNSUPPORTED;  // multi-kernel engine only
        if (!A || A->fmt != GK_CSR || A->n != A->ncols || A->dtype != As[0]->dtype ||
            A->n > 16384 || (A->n > 0 && (!bs[i] || !xs[i])))
            return GK_ERR_INVALID;
        if (A->device != dev) return GK_ERR_UNSUPPORTED;
    }
    cudaStream_t s = (cudaStream_t)stream;
    int32_t nmax = 0;
    for (int32_t i = 0; i < count; ++i) nmax = std::max(nmax, As[i]->n);
    BatchCfg cfg;  // untuned default: CSR
    cfg.nt = nmax > WIDE_BLOCK_ROWS ? 512 : 256;
    int nt = 0;
    if (const char* e = getenv("GK_BATCH_THREADS")) nt = atoi(e);
    const bool fnt = nt == 128 || nt == 256 || nt == 512;
    const bool flay = forced_layout(&cfg);
    const char* at = getenv("GK_AUTOTUNE");
    // batches of fewer than TUNE_MIN_COUNT systems run the untuned default:
    // their trial runs cost more than a better layout saves (the serving
    // loop's varying small batches, each a new shape, lost ~20 % of their
    // throughput to them: 81 against 100 solves/s at saturation)
    if (!(fnt && flay) && !(at && at[0] == '0') && count >= TUNE_MIN_COUNT) {
        const uint64_t key = tune_key(As[0]->dtype, o, nmax, count);
        bool found = false;
        BatchCfg tuned;
        {
            std::lock_guard<std::mutex> lk(g_tune_mu);
            auto it = g_tune.find(key);
            if (it != g_tune.end()) {
                tuned = it->second;
                found = true;
            }
        }
        if (!found) {
            GK_TRY(autotune(count, As, bs, xs, o, s, &tuned));
            std::lock_guard<std::mutex> lk(g_tune_mu);
            g_tune[key] = tuned;
        }
        if (!flay) {
            cfg.layout = tuned.layout;
            cfg.S = tuned.S;
        }
        if (!fnt) cfg.nt = tuned.nt;
    }
    if (fnt) cfg.nt = nt;
    return run_batch(count, As, bs, xs, o, infos, s, cfg, nullptr);
}
