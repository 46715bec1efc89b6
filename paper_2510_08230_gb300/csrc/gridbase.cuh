// gridbase.cuh - what the persistent grid-wide solvers (gridcg.cuh, gridgm.cuh)
// share: blocks of one cooperative launch that own contiguous rows of an ELL
// matrix, sum over the grid and publish the gathered vector.
//
// Hand-off of a reduction: every block posts its partial sums to slots of
// its own, and every block polls all slots, adds them in one fixed order and
// forms the scalars, so all blocks take identical decisions and results do
// not depend on timing.  A slot holding SLOT_EMPTY has not been posted yet:
// value and signal travel in one 8-byte exchange, and no fence is needed
// because no data is handed over with it.  Measured on 152 blocks, cycles from
// post to all seen: exchange 1,700, relaxed store 2,000 to 2,700, a master
// block that collects and rebroadcasts 4,500, clusters of 8 or 16 with one
// poller each 4,400; with a release fence (the gathered vector published): a
// counter 2,500, stores 4,300.  Slots come in three rounds (a publication
// ends a round); a block empties its slots of round k + 1 before it publishes
// in round k: by then every block has left round k - 2, which used them.
// Every poll is bounded by the solve's wait budget.  A wait can run out
// although no block is lost: other work may hold an SM that a block of the
// grid still needs.  Then every block leaves, the error word tells the host
// (a block that had finished does not know), the caller's x is untouched and
// the multi-kernel engine, whose kernels wait for nothing, solves instead.
//
// FP64: a warp instruction holds its sub-partition's pipe for 65 cycles
// whatever its mask (16 cycles of the SM with all four busy), so block sums
// are spread over the sub-partitions and scalars are formed by one lane.
#pragma once

#include "grid_limits.h"
#include "grid_seats.h"
#include "solve_engine.cuh"

namespace gk {

constexpr unsigned long long SLOT_EMPTY = ~0ull;
constexpr int GRID_POLLS = 5;  // slots per polling lane
constexpr int GRID_MAX_BLOCKS = 32 * GRID_POLLS;
template <int NT>
constexpr size_t GRID_RED = 2 * (NT / 2) * sizeof(double);  // scratch of GridTeam::sum
constexpr int GRID_VALUES = 4;  // scalar slots a block and round: 2 sums of up to 2 values
constexpr int GRID_ROUNDS = 3;
constexpr int GRID_CH = 8;     // entries of a row in flight
// Chunks of GRID_CH entries fetched into L2 ahead of their use: a
// whole pass of the block's rows ahead is more than L2 holds when rows are
// wide (121 entries a row, n = 500,000, CG: 203 us per iteration with a
// whole pass, 186 with 4, 155 with 2; 7 entries a row: the same).
constexpr int GRID_AHEAD = 2;
// Threads of a block.  Full: one block an SM; with 32 warps its FP64 pipe
// always finds one whose loads have landed.  Half: two blocks an SM, which
// two solves at once can share (one's arithmetic runs in the other's waits).
// Both at 64 registers a thread.
constexpr int GRID_FULL = 1024, GRID_HALF = 512;
// The half size up to these rows a block, where the vectors fit (CG in FP64
// to 3,400 rows a block, n = 520,000; FP32 to 1,000,000).  Alone (FP64, us per
// iteration of Jacobi-CG and step of Jacobi-GMRES(30), full / half): n = 17,030
// 8.8 / 8.2 and 46.9 / 35.9, 117,453 12.3 / 12.3 and 57.3 / 49.7, 300,763 18.1 /
// 17.9 and 86 / 76, 512,000 24.9 / 25.5 and 113 / 112; with 33 entries a row
// 300,000 36.7 / 41.0 and 110 / 113, with 121 entries a row 90 / 106 and 171 /
// 208 (multi-kernel 154 and 202); FP32 CG 10^6 18.2 / 22.9 (34.7).  What a lone
// solve loses there, a serving mix (24 matrices of 1e3 to 1e6 rows, six
// workers) gains: solves per second at saturation, and p50 / p99 in ms at 0.8
// of it: multi-kernel 100, 103 / 966; half to 2,048 rows and 32,768 entries
// 96, 111 / 619; to 4,096 rows 104, 114 / 694; to 8,192 111, 65 / 618.  GMRES
// takes the half size where it is not the slower one alone.
constexpr int64_t GRID_HALF_ROWS = 8192;
constexpr int64_t GRID_GM_HALF_ROWS = 4096, GRID_GM_HALF_ENTRIES = 131072;
// The least rows of a block, in bytes of a vector: fewer blocks leave SMs to
// other solves and make the hand-offs cheaper.  Six solves of 17K to 25K rows
// at once, 64 / 256 / 512 rows a block: FP64 CG 17.6 / 12.0 / 12.1 ms with
// 8.5 / 8.2 / 8.6 us per iteration alone; inner FP32 solves 16.8 / 11.2 /
// 8.5 ms with 8.0 / 7.4 / 7.4 us.
constexpr int64_t GRID_MIN_ROW_BYTES = 2048;

// GridTeam::between for a budget: below 10 ms the clock is read at every poll.
inline unsigned grid_polls_between(uint64_t wait_ns) { return wait_ns < 10000000 ? 0u : 255u; }

// why a solve ends (0: it goes on); PASSED, CYCLE: a recurrence residual
// passed, a GMRES cycle ended
enum : int { END_OK = 1, END_ZERO, END_INNER, END_CAP, END_NAN, END_BREAKDOWN, END_TIMEOUT, PASSED,
             CYCLE };

struct GridOut {
    int32_t status, iters, restarts, pad;
    double rec, tru;
};

__device__ __forceinline__ int end_status(int end) {
    return end == END_OK || end == END_ZERO || end == END_INNER ? GK_OK
           : end == END_NAN                                     ? GK_ERR_NAN
           : end == END_BREAKDOWN                               ? GK_BREAKDOWN
           : end == END_CAP                                     ? GK_NOT_CONVERGED
                                                                : GK_ERR_TIMEOUT;
}

__device__ __forceinline__ unsigned long long ld_slot(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void post_slot(unsigned long long* p, double v) {
    unsigned long long u = (unsigned long long)__double_as_longlong(v);
    if (u == SLOT_EMPTY) u = 0x7ff8000000000000ull;  // any other NaN
    atomicExch(p, u);
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

// The hand-offs of one block.  slots: [GRID_ROUNDS][GRID_VALUES][nb] then,
// with vectors of nc values, [GRID_ROUNDS][2][nb][nc]; all SLOT_EMPTY, and
// arrived 0, at launch.
template <int NT>
struct GridTeam {
    unsigned long long* slots;
    unsigned long long* arrived;  // blocks that have published, all rounds
    int32_t* err;
    uint64_t wait_ns;
    unsigned between;  // polls between looks at the clock, less 1: 255 or 0
    int nb, nc;
    bool upper;     // threads of the upper half hold values
    double* red;    // shared: GRID_RED<NT> bytes
    double* part;   // shared: 8 values
    int* code;      // shared
    unsigned round;

    __device__ __forceinline__ unsigned long long* slot(unsigned rd, int v) const {
        return slots + ((size_t)(rd % GRID_ROUNDS) * GRID_VALUES + v) * nb;
    }
    __device__ __forceinline__ unsigned long long* vslot(unsigned rd, int which) const {
        return slots + (size_t)GRID_ROUNDS * GRID_VALUES * nb +
               ((size_t)(rd % GRID_ROUNDS) * 2 + which) * nb * nc;
    }

    // A warp spins until ready() holds in all lanes; false: the budget ran
    // out, here or elsewhere.  The clock is read every 256 polls (one of ~700
    // cycles), or with a budget that this would overrun at every poll.
    template <class F>
    __device__ __forceinline__ bool wait(F&& ready) const {
        uint64_t t0 = 0;
        // counts in steps of 1, or 256, so that the test is against a constant
        // (a mask of the budget's: 117,000-row CG 3.16 ms, so 2.94; 128^3 42.6
        // and 42.5)
        for (unsigned spin = 255u - between;; spin += 256u - between) {
            if (__all_sync(0xffffffffu, ready())) return true;
            if ((spin & 255u) != 255u) continue;
            bool stop = false;
            if ((threadIdx.x & 31) == 0) {
                const uint64_t t = globaltimer_ns();
                if (t0 == 0) t0 = t;
                stop = t - t0 > wait_ns || *reinterpret_cast<volatile int32_t*>(err) != 0;
                if (stop) atomicExch(err, 1);
            }
            if (__any_sync(0xffffffffu, stop)) return false;
        }
    }

    // Sums NA values over the grid, runs fin(totals) on one lane (which
    // leaves what follows from them in shared memory) and returns its code in
    // every thread.  kind 0 and 1: each at most once a round.  The block's
    // tree: one add for the upper half of the threads, then four warps add
    // PER values a lane and shuffle.
    template <int NA, class Fin>
    __device__ __forceinline__ int sum(int kind, const double* v, Fin&& fin) {
        constexpr int HT = NT / 2, PER = HT / 128;  // values a lane of the four warps adds
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
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
            const double* w = red + warp * 32 * PER + lane;
            auto lane_sum = [&] { return PER == 4 ? (w[0] + w[32]) + (w[64] + w[96]) : w[0] + w[32]; };
            static_assert(PER == 4 || PER == 2, "full and half blocks");
            const double t0 = lane_sum();
            if constexpr (NA == 2) {
                w += HT;
                const double t = warp_sum2(t0, lane_sum());
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
                post_slot(slot(round, 2 * kind + lane) + blockIdx.x, (w[0] + w[1]) + (w[2] + w[3]));
            }
            const unsigned long long* sl = slot(round, 2 * kind);
            unsigned long long u[NA][GRID_POLLS];
            const bool ok = wait([&] {
                bool all = true;
#pragma unroll
                for (int a = 0; a < NA; ++a)
#pragma unroll
                    for (int j = 0; j < GRID_POLLS; ++j) {
                        const int i = lane + 32 * j;
                        u[a][j] = i < nb ? ld_slot(sl + (size_t)a * nb + i) : 0ull;
                    }
#pragma unroll
                for (int a = 0; a < NA; ++a)
#pragma unroll
                    for (int j = 0; j < GRID_POLLS; ++j) all &= u[a][j] != SLOT_EMPTY;
                return all;
            });
            double tot[NA];
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                double x[GRID_POLLS];
#pragma unroll
                for (int j = 0; j < GRID_POLLS; ++j) x[j] = __longlong_as_double((long long)u[a][j]);
                tot[a] = ((x[0] + x[1]) + (x[2] + x[3])) + x[4];
            }
            if constexpr (NA == 2) {
                tot[0] = warp_sum2(tot[0], tot[1]);
                tot[1] = __shfl_sync(0xffffffffu, tot[0], 16);
            } else {
                tot[0] = warp_sum(tot[0]);
            }
            if (lane == 0) *code = ok ? fin(tot) : END_TIMEOUT;
        }
        __syncthreads();
        return *code;
    }
    static_assert(GRID_POLLS == 5, "sum adds five polled values a lane");

    // Ends a round: everything this block wrote to the gathered vector is
    // visible to every block afterwards.  False: a wait ran out.
    __device__ __forceinline__ bool publish() {
        const int tid = threadIdx.x;
        for (int i = tid; i < GRID_VALUES + 2 * nc; i += NT) {
            if (i < GRID_VALUES) {
                *(slot(round + 1, i) + blockIdx.x) = SLOT_EMPTY;
            } else {
                const int which = i - GRID_VALUES >= nc, c = i - GRID_VALUES - which * nc;
                vslot(round + 1, which)[(size_t)blockIdx.x * nc + c] = SLOT_EMPTY;
            }
        }
        __syncthreads();
        ++round;
        if (tid < 32) {
            if (tid == 0) {
                __threadfence();
                atomicAdd(arrived, 1ull);
            }
            const unsigned long long want = (unsigned long long)round * nb;
            const bool ok = wait([&] { return tid != 0 || ld_slot(arrived) >= want; });
            __threadfence();
            if (tid == 0) *code = ok ? 0 : -1;
        }
        __syncthreads();
        return *code == 0;
    }
};

// The block's rows [r0, r0 + nloc) of an ELL matrix, in shared memory (STAGED:
// entry j of row li at j R + li) or in global memory.
template <int NT, typename V, typename T, bool STAGED>
struct GridRows {
    int32_t R, K, r0, nloc;
    int64_t stride;
    const int32_t* col;
    const V* val;
    V* s_val;        // shared
    int32_t* s_col;  // shared

    __device__ __forceinline__ void stage() const {
        if constexpr (STAGED)
            for (int32_t j = 0; j < K; ++j)
                for (int32_t li = threadIdx.x; li < nloc; li += NT) {
                    s_val[j * R + li] = val[(int64_t)j * stride + r0 + li];
                    s_col[j * R + li] = col[(int64_t)j * stride + r0 + li];
                }
    }

    // f(li) for every row of this thread (the same rows each time)
    template <class F>
    __device__ __forceinline__ void each(F&& f) const {
#pragma unroll 2
        for (int32_t li = threadIdx.x; li < nloc; li += NT) f(li);
    }

    // Brings GRID_CH entries from `first` on of the 32 rows from li on (a
    // multiple of 32) into L2 while the warp works on others: one lane per
    // 128-byte line, so it costs an instruction or two and no registers.
    __device__ __forceinline__ void prefetch(int32_t li, int32_t first) const {
        constexpr int VL = 32 * (int)sizeof(V) > 128 ? 32 * (int)sizeof(V) / 128 : 1;
        static_assert(GRID_CH * (VL + 1) <= 32, "one line a lane");
        const int k = threadIdx.x & 31, l = k % (VL + 1);
        const int32_t j = first + k / (VL + 1);
        if (STAGED || li >= nloc || k >= GRID_CH * (VL + 1) || j >= K) return;
        const uint32_t at = (uint32_t)j * (uint32_t)stride + (uint32_t)(r0 + li);
        const char* q = l == VL ? reinterpret_cast<const char*>(col) + at * 4u
                                : reinterpret_cast<const char*>(val) + at * (uint32_t)sizeof(V) + 128u * l;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(q));
    }

    // The first entries of the next product's first rows.
    __device__ __forceinline__ void prefetch_first() const {
        for (int32_t j = 0; j < min(K, GRID_AHEAD * GRID_CH); j += GRID_CH) prefetch(threadIdx.x & ~31, j);
    }

    // f(li, sum): the row times the gathered vector p (plain loads: p changes
    // between rounds, and the fences of publish() order them).  Offsets into
    // the matrix are 32-bit bytes (the host checks that they fit).
    template <class F>
    __device__ __forceinline__ void product(const T* p, F&& f) const {
        constexpr int CH = GRID_CH;
        const int32_t wide = (K + CH - 1) / CH * CH;
        const int32_t ahead = min(GRID_AHEAD * CH, wide);
        const uint32_t ld = STAGED ? (uint32_t)R : (uint32_t)stride;
        const char* vals = reinterpret_cast<const char*>(STAGED ? s_val : val);
        const char* cols = reinterpret_cast<const char*>(STAGED ? s_col : col);
        for (int32_t li = threadIdx.x; li < nloc; li += NT) {
            const int32_t li0 = li - (int32_t)(threadIdx.x & 31);
            T s = T(0);
            uint32_t at = STAGED ? (uint32_t)li : (uint32_t)(r0 + li);
            for (int32_t left = K; left > 0; left -= CH, at += CH * ld) {
                const int32_t next = K - left + ahead;
                prefetch(next < wide ? li0 : li0 + NT, next < wide ? next : next - wide);
                int32_t c[CH];
                V v[CH];
                T xv[CH];
#pragma unroll
                for (int u = 0; u < CH; ++u) {
                    c[u] = -1;
                    if (u < left) {
                        const int32_t* q = reinterpret_cast<const int32_t*>(cols + (at + u * ld) * 4u);
                        c[u] = STAGED ? *q : __ldcs(q);
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
    }
};

// ------------------------------------------------------------ host side

// Admission of cooperative grids.  A full block fills an SM and a half block
// half of one (threads and registers; shared memory at most that), so one
// full grid, or half grids of together no more blocks than 2 an SM, are
// resident at once wherever the blocks land: no grid is launched that would
// have to wait for another's blocks.  First come, first served, on each
// device by itself (the current one).
class GridSeats {
public:
    GridSeats(bool half, int blocks);
    ~GridSeats();
    GridSeats(const GridSeats&) = delete;
    GridSeats& operator=(const GridSeats&) = delete;
    float waited_ms = 0.f;  // host time until the seats were free

private:
    SeatPool* pool_;
    int seats_;
};

// Below this GMRES keeps the multi-kernel engine: its steps there are short
// (us, multi-kernel / grid, FP32, m = 30: n = 64 36 / 40, 400 39.5 / 41,
// 1,600 49 / 41; FP64 49 / 45, 52 / 46, 91 / 46).
constexpr int32_t GRID_GMRES_MIN_N = 1024;

// Whether gk_solve's automatic engine may take this solve to a grid kernel.
inline bool grid_admits(gk_matrix M, int method, int pkind) {
    return (method == GK_CG || (method == GK_GMRES && M->n >= GRID_GMRES_MIN_N)) && pkind <= 1 && M->fmt == GK_ELL && M->K > 0 &&
           !getenv("GK_SOLVE_UNROLLED") && !solve_loop_on_host();
}

// The split of a matrix over the blocks, and the hand-offs' device memory.
struct GridPlan {
    int64_t R = 0;  // rows per block
    int nb = 0;     // blocks
    int64_t room[2] = {0, 0};  // dynamic shared memory of a full and of a half block
    bool half = false;
    char* sync = nullptr;
    size_t slot_bytes = 0;
    unsigned long long* slots() const { return (unsigned long long*)sync; }
    unsigned long long* arrived() const { return (unsigned long long*)(sync + slot_bytes); }
    int32_t* err() const { return (int32_t*)(sync + slot_bytes + 128); }
    GridOut* out() const { return (GridOut*)(sync + slot_bytes + 192); }
};

// GK_ERR_UNSUPPORTED: no cooperative launches, or the kernels' 32-bit byte
// offsets do not reach the whole matrix.
inline gk_status grid_plan(gk_matrix M, SolverCache* C, int nc, GridPlan* P) {
    const int sms = std::min(num_sms(), GRID_MAX_BLOCKS);
    P->R = std::max<int64_t>(GRID_MIN_ROW_BYTES / (int64_t)vector_bytes(M->dtype),
                             (((int64_t)M->n + sms - 1) / sms + 63) / 64 * 64);
    P->nb = (int)(((int64_t)M->n + P->R - 1) / P->R);
    int dev = 0, optin = 0, coop = 0;
    GK_CUDA(cudaGetDevice(&dev));
    GK_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    GK_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    // less the kernels' static shared memory, and 1 KB the system keeps of each block
    P->room[0] = (int64_t)optin - 1024;
    P->room[1] = P->R <= GRID_HALF_ROWS ? ((int64_t)optin + 1024) / 2 - 2048 : 0;
    if (!coop || !grid_offsets_fit(M->K, M->stride, (int64_t)value_bytes(M->dtype)))
        return GK_ERR_UNSUPPORTED;
    P->slot_bytes = (sizeof(unsigned long long) * GRID_ROUNDS * (GRID_VALUES + 2 * (size_t)nc) *
                         GRID_MAX_BLOCKS + 255) & ~(size_t)255;
    GK_TRY(C->gsync.ensure(P->slot_bytes + 256));
    P->sync = static_cast<char*>(C->gsync.ptr);
    return GK_OK;
}

// Clears the hand-offs and launches kern(args) on all blocks at once.
template <int NT, typename K, typename A>
gk_status grid_launch(K kern, A& args, const GridPlan& P, size_t smem, cudaStream_t s) {
    GK_TRY(allow_max_dynamic_smem(kern));
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, NT, smem) != cudaSuccess ||
        occ < (NT == GRID_HALF ? 2 : 1) || (int64_t)occ * num_sms() < P.nb) {
        cudaGetLastError();
        return GK_ERR_UNSUPPORTED;
    }
    GK_CUDA(cudaMemsetAsync(P.sync, 0xff, P.slot_bytes, s));
    GK_CUDA(cudaMemsetAsync(P.sync + P.slot_bytes, 0, 256, s));
    void* a[] = {&args};
    const cudaError_t e =
        cudaLaunchCooperativeKernel((const void*)kern, dim3(P.nb), dim3(NT), a, smem, s);
    if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
        cudaGetLastError();
        return GK_ERR_UNSUPPORTED;
    }
    GK_CUDA(e);
    return GK_OK;
}

// x = from when the solve ended by itself: a wait that ran out leaves x alone.
template <typename T>
static __global__ void __launch_bounds__(256)
k_grid_take(int32_t n, const int32_t* __restrict__ err, const GridOut* __restrict__ o,
            const T* __restrict__ from, T* __restrict__ x) {
    if (*err != 0 || o->status == GK_ERR_TIMEOUT) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        x[i] = from[i];
}

// Runs launch() when the GPU has seats for its grid, copies the solution from
// `from` to x and reads the outcome.  The stream is drained first and before
// the seats are given back: they are held for the solve alone.
// GK_ERR_UNSUPPORTED: a wait ran out; x is as it was.
template <typename T, class F>
gk_status grid_run(SolverCache* C, const GridPlan& P, cudaStream_t s, SolveOut* out, int32_t n,
                   const T* from, T* x, F&& launch) {
    struct Outcome {
        int32_t err, pad[15];
        GridOut o;
    };
    static_assert(sizeof(Outcome) <= HDR, "the pinned header holds the outcome");
    Outcome* h = reinterpret_cast<Outcome*>(C->hst);
    GK_CUDA(cudaStreamSynchronize(s));
    {
        GridSeats seats(P.half, P.nb);
        out->queued_ms += seats.waited_ms;
        GK_TRY(launch());
        k_grid_take<T><<<(unsigned)std::min<int64_t>(((int64_t)n + 255) / 256, (int64_t)num_sms() * 8),
                         256, 0, s>>>(n, P.err(), P.out(), from, x);
        GK_CUDA(cudaGetLastError());
        GK_CUDA(cudaMemcpyAsync(h, P.err(), sizeof(Outcome), cudaMemcpyDeviceToHost, s));
        GK_CUDA(cudaStreamSynchronize(s));
    }
    if (h->err != 0 || h->o.status == GK_ERR_TIMEOUT) return GK_ERR_UNSUPPORTED;
    out->threads = P.half ? GRID_HALF : GRID_FULL;
    out->status = (gk_status)h->o.status;
    out->iters = h->o.iters;
    out->restarts = h->o.restarts;
    out->rec = h->o.rec;
    out->tru = h->o.tru;
    return GK_OK;
}

// The kernels' vectors; GK_ERR_UNSUPPORTED when there is no room for them
// (the handle may hold the multi-kernel engine's already).
inline gk_status grid_vectors(SolverCache* C, size_t bytes) {
    const gk_status st = C->gvecs.ensure(bytes);
    if (st != GK_ERR_OOM) return st;
    cudaGetLastError();
    return GK_ERR_UNSUPPORTED;
}

}  // namespace gk
