// matrix.cu - matrix handles: creation (CSR, COO), validation, format and
// value-type conversion, export, launch planning.
//
// COO -> CSR follows the ordering rule of the library's COO entry point:
// entries sorted by (row, col); equal (row, col) entries summed in input
// order; explicit zeros kept.  The device algorithm is: count rows, scan,
// scatter (row, col, input position) keys into row buckets in any order,
// sort each bucket by (col, input position) - a total order, so the result
// does not depend on the scatter order - then merge equal columns left to
// right.  Sorting goes by classes of row length, merging by entries, so that
// neither waits for one long row.
#include <algorithm>
#include <cstring>
#include <vector>

#include <shared_mutex>

#include "spmv.cuh"

namespace gk {

static thread_local std::string g_last_error;

void set_error(const char* where, cudaError_t e) {
    g_last_error = std::string(where) + ": " + cudaGetErrorString(e);
}
const char* last_error() { return g_last_error.c_str(); }

static std::shared_mutex g_gate;
static thread_local int g_gate_depth = 0;   // shared holds of this thread
static thread_local bool g_in_capture = false;

GateShared::GateShared() : held(false) {
    if (g_in_capture) return;
    if (g_gate_depth++ == 0) {
        g_gate.lock_shared();
        held = true;
    }
}
GateShared::~GateShared() {
    if (g_in_capture) return;
    if (--g_gate_depth == 0 && held) g_gate.unlock_shared();
}
GateCapture::GateCapture() {
    g_gate.lock();
    g_in_capture = true;
}
GateCapture::~GateCapture() {
    g_in_capture = false;
    g_gate.unlock();
}

cudaError_t dmalloc(void** p, size_t bytes) {
    GateShared gate;
    *p = nullptr;
    return cudaMalloc(p, bytes + 64);
}
void dfree(void* p) {
    GateShared gate;
    if (p) cudaFree(p);
}

gk_status DevBuf::ensure(size_t want) {
    if (want <= bytes && ptr) return GK_OK;
    GateShared gate;
    if (ptr) {
        cudaFree(ptr);
        ptr = nullptr;
        bytes = 0;
    }
    size_t b = std::max<size_t>(want, 256);
    GK_CUDA(dmalloc(&ptr, b));
    bytes = b;
    return GK_OK;
}
void DevBuf::release() {
    GateShared gate;
    if (ptr) cudaFree(ptr);
    ptr = nullptr;
    bytes = 0;
}

int num_sms() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    return sms;
}

__global__ void k_scan_blocksums(int64_t* __restrict__ bsum, int64_t nb) {
    __shared__ int64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < nb; base += SCAN_TILE) {
        int64_t v[SCAN_ITEMS];
        const int64_t my = base + (int64_t)threadIdx.x * SCAN_ITEMS;
#pragma unroll
        for (int i = 0; i < SCAN_ITEMS; ++i) v[i] = (my + i < nb) ? bsum[my + i] : 0;
        int64_t tot = block_excl_scan(v);
        const int64_t c = carry;
#pragma unroll
        for (int i = 0; i < SCAN_ITEMS; ++i)
            if (my + i < nb) bsum[my + i] = v[i] + c;
        __syncthreads();
        if (threadIdx.x == 0) carry = c + tot;
        __syncthreads();
    }
}

// ---------------------------------------------------------------- kernels

// Validation of a CSR copy.  err bits: 1 row_ptr[0] != 0, 2 decreasing,
// 4 row_ptr[n] != nnz, 8 column out of range.  Also the longest row and the
// number of empty rows.
__global__ void k_validate_rowptr(int32_t n, int64_t nnz, const int32_t* __restrict__ rp,
                                  unsigned int* err, int32_t* max_row, int32_t* n_empty) {
    int32_t local_max = 0, local_empty = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t a = rp[i], b = rp[i + 1];
        if (b < a) atomicOr(err, 2u);
        else local_max = max(local_max, b - a);
        local_empty += b == a;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (rp[0] != 0) atomicOr(err, 1u);
        if ((int64_t)rp[n] != nnz) atomicOr(err, 4u);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) local_max = max(local_max, __shfl_xor_sync(0xffffffffu, local_max, o));
    if ((threadIdx.x & 31) == 0 && local_max > 0) atomicMax(max_row, local_max);
    local_empty = __reduce_add_sync(0xffffffffu, local_empty);
    if ((threadIdx.x & 31) == 0 && local_empty > 0) atomicAdd(n_empty, local_empty);
}

__global__ void k_validate_cols(int64_t nnz, int32_t ncols, const int32_t* __restrict__ ci,
                                unsigned int* err) {
    bool bad = false;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nnz;
         k += (int64_t)gridDim.x * blockDim.x) {
        int32_t c = ci[k];
        bad |= (c < 0) | (c >= ncols);
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(err, 8u);
}

// Counts the entries of every row; rank[k] = entry k's place among its row's
// in arrival order (any order: the rows are sorted).
__global__ void k_coo_count(int64_t nnz, int32_t n, int32_t ncols, const int32_t* __restrict__ row,
                            const int32_t* __restrict__ col, int32_t* __restrict__ cnt,
                            int32_t* __restrict__ rank, unsigned int* err) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nnz;
         k += (int64_t)gridDim.x * blockDim.x) {
        int32_t r = row[k], c = col[k];
        if (r < 0 || r >= n || c < 0 || c >= ncols) {
            atomicOr(err, 8u);
            continue;
        }
        rank[k] = atomicAdd(cnt + r, 1);
    }
}

__global__ void k_coo_scatter(int64_t nnz, const int32_t* __restrict__ row,
                              const int32_t* __restrict__ col, const int32_t* __restrict__ start,
                              const int32_t* __restrict__ rank, uint64_t* __restrict__ keys) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nnz;
         k += (int64_t)gridDim.x * blockDim.x)
        keys[start[row[k]] + rank[k]] = ((uint64_t)(uint32_t)col[k] << 32) | (uint64_t)(uint32_t)k;
}

// Rows are sorted by classes of length, each with its own kernel and list of
// rows (a kernel that visits every row to find its own spends most of its
// lanes on others'): classes 0 to 8 hold lengths 2, ..4, ..8, up to ..512 (a
// group of 2 to 32 lanes, then a warp with 2 to 16 keys a lane), 9 lengths to
// SORT_BLOCK_MAX (a block), 10 longer ones.  Rows of one entry need none.
constexpr int SORT_CLASSES = 11;
constexpr int SORT_BLOCK_MAX = 16384;  // keys in shared memory (128 KB)

__device__ __forceinline__ int sort_class(int32_t L) {
    if (L < 2) return -1;
    if (L > 512) return L <= SORT_BLOCK_MAX ? 9 : 10;
    return 31 - __clz(L - 1);  // 2: 0, 3-4: 1, 5-8: 2, ... 257-512: 8
}

// Sizes of the classes and the longest row ({sizes, longest} in `out`).
__global__ void k_class_sizes(int32_t n, const int32_t* __restrict__ cnt, int32_t* __restrict__ out) {
    __shared__ int32_t sz[SORT_CLASSES + 1];
    if (threadIdx.x <= SORT_CLASSES) sz[threadIdx.x] = 0;
    __syncthreads();
    int32_t longest = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t L = cnt[i];
        const int c = sort_class(L);
        if (c >= 0) atomicAdd(sz + c, 1);
        longest = max(longest, L);
    }
    atomicMax(sz + SORT_CLASSES, longest);
    __syncthreads();
    if (threadIdx.x < SORT_CLASSES && sz[threadIdx.x]) atomicAdd(out + threadIdx.x, sz[threadIdx.x]);
    if (threadIdx.x == SORT_CLASSES) atomicMax(out + SORT_CLASSES, sz[SORT_CLASSES]);
}

struct ClassOffsets {
    int32_t o[SORT_CLASSES];
};

// Lists the rows of every class (in any order) from off.o[class] on.
__global__ void k_class_lists(int32_t n, const int32_t* __restrict__ cnt, ClassOffsets off,
                              int32_t* __restrict__ cursor, int32_t* __restrict__ list) {
    __shared__ int32_t sz[SORT_CLASSES], base[SORT_CLASSES];
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (threadIdx.x < SORT_CLASSES) sz[threadIdx.x] = 0;
    __syncthreads();
    const int c = i < n ? sort_class(cnt[i]) : -1;
    const int32_t at = c >= 0 ? atomicAdd(sz + c, 1) : 0;
    __syncthreads();
    if (threadIdx.x < SORT_CLASSES && sz[threadIdx.x])
        base[threadIdx.x] = off.o[threadIdx.x] + atomicAdd(cursor + threadIdx.x, sz[threadIdx.x]);
    __syncthreads();
    if (c >= 0) list[base[c] + at] = (int32_t)i;
}

// Rows of length in (W/2, W] (W <= 32): W-lane bitonic networks.
template <int W>
__global__ void k_sort_rows_sub(int32_t m, const int32_t* __restrict__ list,
                                const int32_t* __restrict__ start, uint64_t* __restrict__ keys) {
    const int lane = threadIdx.x & (W - 1);
    const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / W;
    const int64_t ng = ((int64_t)gridDim.x * blockDim.x) / W;
    // the loop trip count is uniform across the warp (groups advance together)
    const int64_t warp_first = g - (threadIdx.x & 31) / W;
    for (int64_t base = warp_first; base < m; base += ng) {
        const int64_t q = base + (threadIdx.x & 31) / W;
        int32_t a = 0, L = 0;
        if (q < m) {
            const int32_t r = list[q];
            a = start[r];
            L = start[r + 1] - a;
        }
        uint64_t v = lane < L ? keys[a + lane] : ~0ull;
#pragma unroll
        for (int k = 2; k <= W; k <<= 1) {
#pragma unroll
            for (int j = k >> 1; j > 0; j >>= 1) {
                uint64_t o = __shfl_xor_sync(0xffffffffu, v, j, W);
                bool up = ((lane & k) == 0);
                bool lower = ((lane & j) == 0);
                uint64_t mn = v < o ? v : o, mx = v < o ? o : v;
                v = (lower == up) ? mn : mx;
            }
        }
        if (lane < L) keys[a + lane] = v;
    }
}

// Bitonic exchanges of 32 E keys in a warp's registers, key i in register
// i / 32 of lane i mod 32: those over 32 and more places stay in a lane.
// One step of distance j of the merge of size k; `down`: the order of keys
// whose bit k is clear is descending.
template <int E>
__device__ __forceinline__ void bitonic_step(uint64_t (&v)[E], int k, int j, bool down) {
    const int lane = threadIdx.x & 31;
    if (j >= 32) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int f = e ^ (j >> 5);
            if (f > e) {
                const bool up = (((e << 5) & k) == 0) != down;
                const uint64_t x = v[e], y = v[f];
                const bool swap = (x > y) == up;
                v[e] = swap ? y : x;
                v[f] = swap ? x : y;
            }
        }
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint64_t o = __shfl_xor_sync(0xffffffffu, v[e], j);
            const bool up = ((((e << 5) | lane) & k) == 0) != down;
            const bool lower = (lane & j) == 0;
            v[e] = (lower == up) == (v[e] < o) ? v[e] : o;
        }
    }
}

// Sorts the 32 E keys, ascending or (last_down) descending.
template <int E>
__device__ __forceinline__ void bitonic_sort(uint64_t (&v)[E], bool last_down) {
#pragma unroll
    for (int k = 2; k <= 32 * E; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) bitonic_step<E>(v, k, j, k == 32 * E && last_down);
}

// The steps of distance 16 E and less of a merge larger than the keys.
template <int E>
__device__ __forceinline__ void bitonic_merge(uint64_t (&v)[E], bool down) {
#pragma unroll
    for (int j = 16 * E; j > 0; j >>= 1) bitonic_step<E>(v, 0, j, down);
}

// Rows of length in (16 E, 32 E]: one warp each.
template <int E>
__global__ void __launch_bounds__(128)
k_sort_rows_warp(int32_t m, const int32_t* __restrict__ list, const int32_t* __restrict__ start,
                 uint64_t* __restrict__ keys) {
    const int lane = threadIdx.x & 31;
    for (int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; q < m;
         q += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int32_t r = list[q], a = start[r], L = start[r + 1] - a;
        uint64_t v[E];
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = e * 32 + lane < L ? keys[a + e * 32 + lane] : ~0ull;
        bitonic_sort<E>(v, false);
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (e * 32 + lane < L) keys[a + e * 32 + lane] = v[e];
    }
}

// Longer rows: one block per row, keys padded to a power of two P in shared
// memory.  Each warp sorts chunks of 512 keys in its registers; of the merge
// steps only the exchanges over 512 and more places go through shared memory
// with a block barrier each (6 of the 78 steps of 4096 keys), the rest of
// every merge runs chunk by chunk in registers again.  2,500 rows of 513 to
// 4096 entries: 215 us, 425 with every step in shared memory.
constexpr int CHUNK_E = 16, CHUNK = 32 * CHUNK_E;

__global__ void __launch_bounds__(256)
k_sort_rows_block(int32_t m, const int32_t* __restrict__ list, const int32_t* __restrict__ start,
                  uint64_t* __restrict__ keys) {
    extern __shared__ uint64_t sk[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int64_t q = blockIdx.x; q < m; q += gridDim.x) {
        const int32_t r = list[q], a = start[r], L = start[r + 1] - a;
        int P = CHUNK;
        while (P < L) P <<= 1;
        for (int base = warp * CHUNK; base < P; base += nw * CHUNK) {
            uint64_t v[CHUNK_E];
#pragma unroll
            for (int e = 0; e < CHUNK_E; ++e) {
                const int i = base + e * 32 + lane;
                v[e] = i < L ? keys[a + i] : ~0ull;
            }
            bitonic_sort<CHUNK_E>(v, (base & CHUNK) != 0);
#pragma unroll
            for (int e = 0; e < CHUNK_E; ++e) sk[base + e * 32 + lane] = v[e];
        }
        __syncthreads();
        for (int k = 2 * CHUNK; k <= P; k <<= 1) {
            for (int j = k >> 1; j >= CHUNK; j >>= 1) {
                for (int t = threadIdx.x; t < P / 2; t += blockDim.x) {
                    const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1)), p = i | j;
                    const bool up = (i & k) == 0;
                    const uint64_t x = sk[i], y = sk[p];
                    if ((x > y) == up) {
                        sk[i] = y;
                        sk[p] = x;
                    }
                }
                __syncthreads();
            }
            for (int base = warp * CHUNK; base < P; base += nw * CHUNK) {
                uint64_t v[CHUNK_E];
#pragma unroll
                for (int e = 0; e < CHUNK_E; ++e) v[e] = sk[base + e * 32 + lane];
                bitonic_merge<CHUNK_E>(v, (base & k) != 0);
#pragma unroll
                for (int e = 0; e < CHUNK_E; ++e) sk[base + e * 32 + lane] = v[e];
            }
            __syncthreads();
        }
        for (int i = threadIdx.x; i < L; i += blockDim.x) keys[a + i] = sk[i];
        __syncthreads();
    }
}

// Rows longer than the shared-memory sorter: bitonic sort in a global
// scratch area of P keys per block.
__global__ void k_sort_rows_global(int32_t m, const int32_t* __restrict__ list,
                                   const int32_t* __restrict__ start, uint64_t* __restrict__ keys,
                                   uint64_t* __restrict__ scratch, int64_t P) {
    uint64_t* sk = scratch + (int64_t)blockIdx.x * P;
    for (int64_t row = blockIdx.x; row < m; row += gridDim.x) {
        const int32_t r = list[row];
        const int64_t a = start[r], L = start[r + 1] - a;
        int64_t Q = 1;
        while (Q < L) Q <<= 1;
        for (int64_t i = threadIdx.x; i < Q; i += blockDim.x) sk[i] = i < L ? keys[a + i] : ~0ull;
        __syncthreads();
        for (int64_t k = 2; k <= Q; k <<= 1) {
            for (int64_t j = k >> 1; j > 0; j >>= 1) {
                for (int64_t i = threadIdx.x; i < Q; i += blockDim.x) {
                    int64_t p = i ^ j;
                    if (p > i) {
                        bool up = ((i & k) == 0);
                        uint64_t x = sk[i], y = sk[p];
                        if ((x > y) == up) {
                            sk[i] = y;
                            sk[p] = x;
                        }
                    }
                }
                __syncthreads();
            }
        }
        for (int64_t i = threadIdx.x; i < L; i += blockDim.x) keys[a + i] = sk[i];
        __syncthreads();
    }
}

// first[p] = 1 where a row begins
__global__ void k_row_firsts(int32_t n, const int32_t* __restrict__ start,
                             unsigned char* __restrict__ first) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n;
         r += (int64_t)gridDim.x * blockDim.x)
        if (start[r + 1] > start[r]) first[start[r]] = 1;
}

// Whether sorted entry p is the first of its (row, col): the others are added
// to it.  The passes below give every entry to a thread, so the time does
// not depend on how the entries spread over the rows (a thread per row took
// 1,634 us for 8M entries, 4096 of them in one row).
__device__ __forceinline__ bool is_head(const uint64_t* __restrict__ keys,
                                        const unsigned char* __restrict__ first, int64_t p) {
    return first[p] || (uint32_t)(keys[p] >> 32) != (uint32_t)(keys[p - 1] >> 32);
}

__global__ void __launch_bounds__(SCAN_THREADS)
k_head_counts(int64_t nnz, const uint64_t* __restrict__ keys,
              const unsigned char* __restrict__ first, int64_t* __restrict__ bsum) {
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    int32_t c = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const int64_t p = base + i * SCAN_THREADS + threadIdx.x;
        if (p < nnz) c += is_head(keys, first, p);
    }
    __shared__ int32_t sh[32];
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x < 32) {
        c = __reduce_add_sync(0xffffffffu, sh[threadIdx.x]);
        if (threadIdx.x == 0) bsum[blockIdx.x] = c;
    }
}

// Writes the heads' columns and sums (each with the equal entries that follow
// it, in input order) at their places, and every entry's number of heads
// before it.  boff: exclusive scan of k_head_counts.
template <typename VIn, typename VOut, typename Acc>
__global__ void __launch_bounds__(SCAN_THREADS)
k_merge_heads(int64_t nnz, const uint64_t* __restrict__ keys,
              const unsigned char* __restrict__ first, const int64_t* __restrict__ boff,
              const VIn* __restrict__ val, int32_t* __restrict__ before,
              int32_t* __restrict__ out_col, VOut* __restrict__ out_val) {
    __shared__ int32_t wsum[SCAN_ITEMS][32], slice[SCAN_ITEMS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    bool head[SCAN_ITEMS];
    unsigned heads[SCAN_ITEMS];
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const int64_t p = base + i * SCAN_THREADS + threadIdx.x;
        head[i] = p < nnz && is_head(keys, first, p);
        heads[i] = __ballot_sync(0xffffffffu, head[i]);
        if (lane == 0) wsum[i][warp] = __popc(heads[i]);
    }
    __syncthreads();
    if (warp < SCAN_ITEMS) {  // exclusive over the warps of slice `warp`
        const int32_t w = wsum[warp][lane];
        const int32_t inc = warp_incl_scan(w);
        wsum[warp][lane] = inc - w;
        if (lane == 31) slice[warp] = inc;
    }
    __syncthreads();
    int64_t o = boff[blockIdx.x];
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const int64_t p = base + i * SCAN_THREADS + threadIdx.x;
        const int32_t at = (int32_t)o + wsum[i][warp] + __popc(heads[i] & ((1u << lane) - 1u));
        if (p < nnz) before[p] = at;
        if (head[i]) {
            const uint64_t key = keys[p];
            Acc s = (Acc)to_acc(val[(uint32_t)key]);
            for (int64_t j = p + 1; j < nnz && !is_head(keys, first, j); ++j)
                s = s + (Acc)to_acc(val[(uint32_t)keys[j]]);
            out_col[at] = (int32_t)(key >> 32);
            out_val[at] = from_acc<VOut>(s);
        }
        o += slice[i];
    }
}

// row_ptr from the entries' counts of heads before them
__global__ void k_row_ptr(int32_t n, int64_t nnz, const int32_t* __restrict__ start,
                          const int32_t* __restrict__ before, const int64_t* __restrict__ total,
                          int32_t* __restrict__ rp) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r <= n;
         r += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = start[r];
        rp[r] = a < nnz ? before[a] : (int32_t)*total;
    }
}

// value conversion (round to nearest even on narrowing)
template <typename VIn, typename VOut>
__global__ void k_convert_values(int64_t m, const VIn* __restrict__ in, VOut* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = cvt<VOut>(in[i]);
}

template <typename VIn, typename VOut>
__global__ void k_csr_to_ell(int32_t n, int64_t stride, int32_t K, const int32_t* __restrict__ rp,
                             const int32_t* __restrict__ ci, const VIn* __restrict__ va,
                             int32_t* __restrict__ ecol, VOut* __restrict__ eval) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < stride;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t a = 0, L = 0;
        if (i < n) {
            a = rp[i];
            L = rp[i + 1] - a;
        }
        for (int32_t j = 0; j < K; ++j) {
            int64_t at = (int64_t)j * stride + i;
            if (j < L) {
                ecol[at] = ci[a + j];
                eval[at] = cvt<VOut>(va[a + j]);
            } else {
                ecol[at] = -1;
                eval[at] = cvt<VOut>(0.0);
            }
        }
    }
}

__global__ void k_slice_lengths(int32_t n, int32_t S, int32_t f, int32_t nslices,
                                const int32_t* __restrict__ rp, int32_t* __restrict__ slen) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nslices;
         s += (int64_t)gridDim.x * blockDim.x) {
        int32_t m = 0;
        int64_t lo = s * S, hi = lo + S < (int64_t)n ? lo + S : (int64_t)n;
        for (int64_t i = lo; i < hi; ++i) m = max(m, rp[i + 1] - rp[i]);
        slen[s] = ((m + f - 1) / f) * f;
    }
}

template <typename VIn, typename VOut>
__global__ void k_csr_to_sellp(int32_t n, int32_t S, int32_t nslices, const int32_t* __restrict__ rp,
                               const int32_t* __restrict__ ci, const VIn* __restrict__ va,
                               const int32_t* __restrict__ slen, const int64_t* __restrict__ sset,
                               int32_t* __restrict__ scol, VOut* __restrict__ sval) {
    const int64_t slots = (int64_t)nslices * S;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < slots;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = i / S, t = i - s * S;
        int32_t a = 0, L = 0;
        if (i < n) {
            a = rp[i];
            L = rp[i + 1] - a;
        }
        const int64_t base = sset[s];
        const int32_t len = slen[s];
        for (int32_t j = 0; j < len; ++j) {
            int64_t at = (base + j) * S + t;
            if (j < L) {
                scol[at] = ci[a + j];
                sval[at] = cvt<VOut>(va[a + j]);
            } else {
                scol[at] = -1;
                sval[at] = cvt<VOut>(0.0);
            }
        }
    }
}

// ELL / SELL-P back to CSR: count stored (col >= 0) entries per row ...
__global__ void k_padded_row_counts(int32_t n, int fmt, int64_t stride, int32_t K, int32_t S,
                                    const int32_t* __restrict__ slen,
                                    const int64_t* __restrict__ sset,
                                    const int32_t* __restrict__ pcol, int32_t* __restrict__ cnt) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t c = 0;
        if (fmt == GK_ELL) {
            for (int32_t j = 0; j < K; ++j) c += pcol[(int64_t)j * stride + i] >= 0;
        } else {
            const int64_t s = i / S, t = i - s * S;
            for (int32_t j = 0; j < slen[s]; ++j) c += pcol[(sset[s] + j) * S + t] >= 0;
        }
        cnt[i] = c;
    }
}

// ... then copy them in order.
template <typename VIn, typename VOut>
__global__ void k_padded_to_csr(int32_t n, int fmt, int64_t stride, int32_t K, int32_t S,
                                const int32_t* __restrict__ slen, const int64_t* __restrict__ sset,
                                const int32_t* __restrict__ pcol, const VIn* __restrict__ pval,
                                const int32_t* __restrict__ rp, int32_t* __restrict__ ci,
                                VOut* __restrict__ va) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        int64_t o = rp[i];
        if (fmt == GK_ELL) {
            for (int32_t j = 0; j < K; ++j) {
                int64_t at = (int64_t)j * stride + i;
                if (pcol[at] >= 0) {
                    ci[o] = pcol[at];
                    va[o] = cvt<VOut>(pval[at]);
                    ++o;
                }
            }
        } else {
            const int64_t s = i / S, t = i - s * S;
            for (int32_t j = 0; j < slen[s]; ++j) {
                int64_t at = (sset[s] + j) * S + t;
                if (pcol[at] >= 0) {
                    ci[o] = pcol[at];
                    va[o] = cvt<VOut>(pval[at]);
                    ++o;
                }
            }
        }
    }
}

__device__ __forceinline__ int32_t rows_before_nnz(int32_t n, const int32_t* __restrict__ rp,
                                                   int64_t target) {
    int32_t lo = 0, hi = n;  // first row r with row_ptr[r] >= target
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        if ((int64_t)rp[mid] < target) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Row-tile plan: tile c holds the rows whose first nonzero lies in
// [c * chunk, (c + 1) * chunk); its staged range is rounded out to 8 entries.
__global__ void k_tile_desc(int32_t n, const int32_t* __restrict__ rp, int32_t chunk,
                            int32_t ntiles, int4* __restrict__ desc) {
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ntiles;
         c += (int64_t)gridDim.x * blockDim.x) {
        const int32_t r0 = rows_before_nnz(n, rp, c * (int64_t)chunk);
        const int32_t r1 = (c + 1 == ntiles) ? n : rows_before_nnz(n, rp, (c + 1) * (int64_t)chunk);
        const int32_t e0 = r0 < r1 ? rp[r0] : 0, e1 = r0 < r1 ? rp[r1] : 0;
        const int32_t a0 = e0 & ~7;
        const int32_t w = (e1 > e0) ? (((e1 + 7) & ~7) - a0) : 0;
        desc[c] = make_int4(r0, r1, a0, w);
    }
}

// Segmented plan: unit u holds the nonzeros from 256 u on; its first row is
// the first of the m listed rows that ends after that point.
__global__ void k_unit_rows(int32_t m, const int32_t* __restrict__ row_end, int32_t nunits,
                            int32_t* __restrict__ unit_row) {
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u <= nunits;
         u += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = u * SEG_UNIT;
        int32_t lo = 0, hi = m;
        while (lo < hi) {
            const int32_t mid = lo + ((hi - lo) >> 1);
            if ((int64_t)row_end[mid] > k) hi = mid;
            else lo = mid + 1;
        }
        unit_row[u] = lo;
    }
}

// Counts the sampled units (every step-th) whose columns span at most
// `span`.  One warp per unit.
__global__ void k_unit_span(int64_t nnz, int32_t nunits, int32_t step, int32_t span,
                            const int32_t* __restrict__ ci, int32_t* __restrict__ count) {
    const int lane = threadIdx.x & 31;
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t u = w * step;
    if (u >= nunits) return;
    int32_t lo = INT32_MAX, hi = 0;
    for (int64_t k = u * SEG_UNIT + lane; k < min((u + 1) * (int64_t)SEG_UNIT, nnz); k += 32) {
        lo = min(lo, ci[k]);
        hi = max(hi, ci[k]);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0 && hi - lo <= span) atomicAdd(count, 1);
}

__global__ void k_nonempty_flags(int32_t n, const int32_t* __restrict__ rp,
                                 int32_t* __restrict__ flag) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        flag[i] = rp[i + 1] > rp[i];
}

// rank[i]: nonempty rows before row i
__global__ void k_split_rows(int32_t n, const int32_t* __restrict__ rp,
                             const int32_t* __restrict__ rank, int32_t* __restrict__ row_end,
                             int32_t* __restrict__ row_id, int32_t* __restrict__ empty) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = rp[i + 1], q = rank[i];
        if (e > rp[i]) {
            row_end[q] = e;
            row_id[q] = (int32_t)i;
        } else {
            empty[i - q] = (int32_t)i;
        }
    }
}

// ------------------------------------------------------------ host helpers

static unsigned grid_for(int64_t work, int threads = 256) {
    int64_t b = (work + threads - 1) / threads;
    int64_t cap = (int64_t)num_sms() * 16;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (unsigned)b;
}

template <class F>
static gk_status dispatch_dtype(gk_dtype d, F&& f) {
    switch (d) {
        case GK_F64: return f(Types<GK_F64>{});
        case GK_F32: return f(Types<GK_F32>{});
        case GK_BF16: return f(Types<GK_BF16>{});
        case GK_F16: return f(Types<GK_F16>{});
    }
    return GK_ERR_INVALID;
}

static gk_matrix new_handle() {
    gk_matrix A = new (std::nothrow) gk_matrix_s();
    if (A) cudaGetDevice(&A->device);
    return A;
}

static void free_arrays(gk_matrix A) {
    if (A->slab) {
        dfree(A->slab);
    } else {
        for (void* q : {(void*)A->row_ptr, (void*)A->col, A->val, (void*)A->words}) dfree(q);
    }
    A->slab = nullptr;
    A->words = nullptr;
    dfree(A->slice_len);
    dfree(A->slice_set);
    dfree(A->plan.tile_desc);
    for (int32_t* q : {A->plan.unit_row, A->plan.row_end, A->plan.row_id, A->plan.empty_rows})
        dfree(q);
    dfree(A->dinv);
    dfree(A->binv);
    A->binv = nullptr;
    A->binv_bs = 0;
    dfree(A->coo_row);
    dfree(A->empty_rows);
    A->coo_row = A->empty_rows = nullptr;
    delete A->ilu;
    delete A->tri;
    A->ilu = A->tri = nullptr;
    A->row_ptr = A->col = nullptr;
    A->val = nullptr;
    A->slice_len = nullptr;
    A->slice_set = nullptr;
    A->plan = CsrPlan();
    A->dinv = nullptr;
}

// row_ptr, col, val (each with the 64 bytes of slack of an allocation of its
// own) and the handle's words in one allocation: a cudaMalloc or cudaFree
// takes 30 to 90 us of host time, as long as the kernels that fill the arrays.
static gk_status alloc_csr(gk_matrix A) {
    auto up = [](size_t b) { return (b + 64 + 255) & ~(size_t)255; };
    const size_t nz = (size_t)std::max<int64_t>(A->nnz, 1);
    const size_t col = up(4 * ((size_t)A->n + 1)), val = col + up(4 * nz);
    const size_t words = val + up(value_bytes(A->dtype) * nz);
    if (dmalloc(&A->slab, words + 256) != cudaSuccess) return GK_ERR_OOM;
    char* p = static_cast<char*>(A->slab);
    A->row_ptr = (int32_t*)p;
    A->col = (int32_t*)(p + col);
    A->val = p + val;
    A->words = (int32_t*)(p + words);
    return GK_OK;
}

static gk_status ensure_words(gk_matrix A) {
    if (!A->words) GK_CUDA(dmalloc_t(&A->words, 64));
    return GK_OK;
}

static void destroy_handle(gk_matrix A) {
    if (!A) return;
    for (gk_matrix L : A->lowp) destroy_handle(L);
    if (A->solve_fmt != A) destroy_handle(A->solve_fmt);
    free_solver_cache(A);
    free_arrays(A);
    A->stage_in.release();
    A->stage_out.release();
    A->carry.release();
    if (A->side) cudaStreamDestroy(A->side);
    if (A->side2) cudaStreamDestroy(A->side2);
    delete A;
}

// COO view of a CSR handle: the row of every entry, and the list of rows
// without entries (the COO kernel never visits them).
__global__ void k_coo_rows(int32_t n, const int32_t* __restrict__ rp, int32_t* __restrict__ rows,
                           int32_t* __restrict__ empty, unsigned int* __restrict__ n_empty) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = rp[i], b = rp[i + 1];
        for (int32_t k = a; k < b; ++k) rows[k] = (int32_t)i;
        if (a == b) empty[atomicAdd(n_empty, 1u)] = (int32_t)i;  // order of the list is free
    }
}

static gk_status build_coo_view(gk_matrix A, cudaStream_t s) {
    DevBuf cnt, tmp_empty;
    GK_TRY(cnt.ensure(16));
    GK_CUDA(cudaMemsetAsync(cnt.ptr, 0, 16, s));
    GK_CUDA(dmalloc_t(&A->coo_row, (size_t)std::max<int64_t>(A->nnz, 1)));
    GK_TRY(tmp_empty.ensure(4 * (size_t)std::max(A->n, 1)));
    if (A->n > 0)
        k_coo_rows<<<grid_for(A->n), 256, 0, s>>>(A->n, A->row_ptr, A->coo_row,
                                                   (int32_t*)tmp_empty.ptr, (unsigned int*)cnt.ptr);
    GK_CUDA(cudaGetLastError());
    unsigned int ne = 0;
    GK_CUDA(cudaMemcpyAsync(&ne, cnt.ptr, 4, cudaMemcpyDeviceToHost, s));
    GK_CUDA(cudaStreamSynchronize(s));
    A->n_empty = (int32_t)ne;
    if (ne) {
        GK_CUDA(dmalloc_t(&A->empty_rows, (size_t)ne));
        GK_CUDA(cudaMemcpyAsync(A->empty_rows, tmp_empty.ptr, 4 * (size_t)ne, cudaMemcpyDeviceToDevice, s));
        GK_CUDA(cudaStreamSynchronize(s));
    }
    A->coo = 1;
    // triplets per lane: 8 in FP64 (fewer FP64 carry adds per nonzero; 343 us
    // against 366 us for 4 on the 4M-row Zipf matrix), 4 in FP32 (279 us
    // against 291 us)
    A->coo_e = A->dtype == GK_F64 ? 8 : 4;
    if (const char* e = getenv("GK_COO_E")) {
        const int v = atoi(e);
        A->coo_e = (v == 8 || v == 12 || v == 16) ? v : 4;
    }
    return GK_OK;
}

// A segmented unit whose columns span at most this much of x counts as local
// (the L1 that the kernel's shared memory leaves is about 100 KB).
constexpr int64_t LOCAL_COLS_BYTES = 64 * 1024;

// CSR launch plan: row tiles when rows are short, the segmented kernel otherwise.
gk_status build_csr_plan(gk_matrix A, cudaStream_t s) {
    CsrPlan& P = A->plan;
    dfree(P.tile_desc);
    for (int32_t* q : {P.unit_row, P.row_end, P.row_id, P.empty_rows}) dfree(q);
    P = CsrPlan();
    GK_TRY(ensure_words(A));
    P.err = A->words;
    GK_CUDA(cudaMemsetAsync(P.err, 0, 4, s));
    if (A->fmt != GK_CSR || A->n == 0) return GK_OK;
    const double mean = A->mean_row;
    int lanes = 1;
    while (lanes < 32 && lanes < mean) lanes <<= 1;
    P.lanes = lanes;
    // row tiles of ~rows_per_tile rows of mean length; staged capacity
    // covers the chunk plus the longest row plus alignment slack
    // measured on GB300 (256^3 stencil): one staged tile per block with
    // 512-row tiles beats deeper per-block pipelines, because more resident
    // blocks hide the x-gather latency better than prefetching does
    int rows_per_tile = 512;
    if (const char* e = getenv("GK_TILE_ROWS")) rows_per_tile = std::max(32, atoi(e));
    int32_t chunk = (int32_t)std::min<double>(
        8192.0, std::max<double>(512.0, rows_per_tile * std::ceil(std::max(mean, 1.0))));
    chunk = (chunk + 7) & ~7;
    const int64_t cap = (int64_t)chunk + A->max_row + 16;
    // warp tiles (kind 3): 32 * wt_rpl rows per warp, staged capacity of the
    // longest possible tile, one stage per warp by default (measured on
    // GB300, 3D 7-point 256^3 FP64: 1 stage 279 us, 2 stages 367 us, 3 644 us:
    // a smaller ring lets more warps reside, which hides the copy latency
    // better than prefetching within a warp); chosen for short rows of
    // near-uniform length when 8 warps' rings leave room for two blocks per SM
    const int64_t vb = (int64_t)value_bytes(A->dtype);
    int wt_rpl = 2;
    if (const char* e = getenv("GK_WT_RPL")) {
        const int v = atoi(e);
        wt_rpl = (v == 1 || v == 4) ? v : 2;
    }
    const int64_t wt_cap = ((int64_t)32 * wt_rpl * A->max_row + 14 + 7) & ~(int64_t)7;
    int wt_nst = 1;
    if (const char* e = getenv("GK_WT_STAGES")) wt_nst = std::max(1, std::min(4, atoi(e)));
    auto wt_block_bytes = [&](int nst) {
        return (int64_t)WT_WARPS * (((int64_t)nst * wt_cap * (4 + vb) + 8 * nst + 127) & ~(int64_t)127);
    };
    const bool wt_fits = wt_block_bytes(wt_nst) <= WT_SMEM_CAP;
    // The kernel of the fused row epilogues (solver) and, unless P.seg, of
    // gk_apply: 3 warp tiles for short rows of near-uniform length, else 1 row
    // tiles, else (kind 2: longer than 1024) the vector kernel.
    int kind = (A->max_row <= 1024) ? 1 : 2;
    if (wt_fits && wt_block_bytes(wt_nst) <= 112 * 1024 && A->max_row <= 2.0 * mean + 1.0)
        kind = 3;
    // gk_apply runs the segmented kernel wherever warp tiles do not apply.
    // Against row tiles (us, FP64 / FP32; n x mean length, exponential
    // lengths, columns within 2000 of the diagonal): 200,000 x 4: 17.6 / 7.0
    // row tiles, 10.1 / 7.9 segmented; x 16: 70.6 / 26.7, 17.9 / 12.6; 2M x 8:
    // 190 / 75, 71 / 47; 4,000 rows of Zipf lengths: 151 / 39, 6.2 / 5.6.
    P.seg = kind != 3;
    // Small matrices, where a launch is latency: kernels that neither stage
    // nor carry.  Rows of at most 16 entries: one row per thread while one
    // wave of its blocks holds them all (us, FP64 / FP32, against warp tiles:
    // 4,096 rows 2.1 / 1.9 and 3.3 / 2.4, 62,500 2.9 / 2.3 and 3.5 / 2.6; past
    // the wave 90,000 4.3 / 3.1 and 4.6 / 2.7).  Longer rows: the vector
    // kernel up to where the other kernel catches up (n x lanes): against warp
    // tiles FP64 10,000 x 32: 5.7 / 6.1 but 30,000 x 16: 7.0 / 4.1, FP32
    // 3,000 x 32: 1.9 / 3.4 but 30,000 x 16: 2.9 / 2.7; against the segmented
    // kernel FP64 30,000 x 8: 5.8 / 7.4, x 16: 9.3 / 8.8, FP32 30,000 x 32:
    // 6.4 / 8.5, 200,000 x 8: 10.4 / 8.8.  A longest row of more than 24
    // steps waits too long (4,000 Zipf rows: 16.5 / 6.2).
    const int64_t threads = (int64_t)A->n * lanes;
    const int64_t line = vb == 8 ? (P.seg ? 320 : 160) : (P.seg ? 1024 : 256);
    if (A->max_row <= 16 ? A->n <= (int64_t)ROW_THREADS * 8 * num_sms()
                         : threads <= line * 1024 && A->max_row <= 24 * lanes) {
        kind = 0;
        P.seg = 0;
        if (A->max_row <= 16) P.lanes = 1;
    }
    if (const char* force = getenv("GK_CSR_KERNEL")) {
        kind = atoi(force);
        P.seg = kind == 2;
    }
    if (kind == 3 && !wt_fits) kind = 1;
    // a single staged tile must fit in shared memory
    if (kind == 1 && ((cap + 7) & ~7) * (int64_t)(4 + value_bytes(A->dtype)) > 200 * 1024) {
        kind = 2;
        P.seg = 1;
    }
    P.kind = kind;
    P.stages = 1;
    if (const char* e = getenv("GK_ROWTILE_STAGES")) P.stages = std::max(1, std::min(3, atoi(e)));
    if (kind == 3) {
        P.stages = wt_nst;
        P.wt_rpl = wt_rpl;
        P.tile_cap = (int32_t)wt_cap;
    } else if (kind == 1) {
        P.chunk = chunk;
        P.tile_cap = (int32_t)((cap + 7) & ~7);
        P.ntiles = (int32_t)std::max<int64_t>(1, (A->nnz + chunk - 1) / chunk);
        GK_CUDA(dmalloc_t(&P.tile_desc, (size_t)P.ntiles));
        k_tile_desc<<<grid_for(P.ntiles), 256, 0, s>>>(A->n, A->row_ptr, chunk, P.ntiles,
                                                       P.tile_desc);
        GK_CUDA(cudaGetLastError());
    }
    if (P.seg) {
        // units of SEG_UNIT nonzeros over the nonempty rows
        P.units = (int32_t)((A->nnz + SEG_UNIT - 1) / SEG_UNIT);
        TmpBuf flag, rank, tmp;
        int32_t m = A->n;  // nonempty rows
        if (A->empty_rows_known != 0) {
            GK_TRY(flag.ensure(4 * (size_t)A->n));
            GK_TRY(rank.ensure(4 * ((size_t)A->n + 1)));
            int32_t* dflag = static_cast<int32_t*>(flag.ptr);
            int32_t* drank = static_cast<int32_t*>(rank.ptr);
            k_nonempty_flags<<<grid_for(A->n), 256, 0, s>>>(A->n, A->row_ptr, dflag);
            GK_TRY(scan_exclusive<int32_t, int32_t>(dflag, drank, A->n, tmp, s));
            GK_CUDA(cudaMemcpyAsync(&m, drank + A->n, 4, cudaMemcpyDeviceToHost, s));
            GK_CUDA(cudaStreamSynchronize(s));
            P.n_empty = A->n - m;
            if (P.n_empty) {
                GK_CUDA(dmalloc_t(&P.row_end, (size_t)std::max(m, 1)));
                GK_CUDA(dmalloc_t(&P.row_id, (size_t)std::max(m, 1)));
                GK_CUDA(dmalloc_t(&P.empty_rows, (size_t)P.n_empty));
                k_split_rows<<<grid_for(A->n), 256, 0, s>>>(A->n, A->row_ptr, drank, P.row_end,
                                                            P.row_id, P.empty_rows);
                GK_CUDA(cudaStreamSynchronize(s));  // the scratch goes
            }
        }
        // gathers through L1 when most units' columns fit a part of it
        if (P.units > 0) {
            const int32_t step = std::max(1, P.units / 4096);
            const int32_t sampled = (P.units + step - 1) / step;
            int32_t* cnt = A->words + 16;
            GK_CUDA(cudaMemsetAsync(cnt, 0, 4, s));
            k_unit_span<<<(unsigned)((sampled + 7) / 8), 256, 0, s>>>(
                A->nnz, P.units, step, (int32_t)(LOCAL_COLS_BYTES / vector_bytes(A->dtype)), A->col,
                cnt);
            int32_t close = 0;
            GK_CUDA(cudaMemcpyAsync(&close, cnt, 4, cudaMemcpyDeviceToHost, s));
            GK_CUDA(cudaStreamSynchronize(s));
            P.local_cols = 2 * close > sampled;
        }
        const size_t urow = (4 * ((size_t)P.units + 1) + 255) & ~(size_t)255;
        P.slots = A->max_row > SEG_HEADS_MAX ? 1 : StreamSlots::COUNT;
        P.carry_bytes = ((size_t)P.units * (4 + vector_bytes(A->dtype)) + 16 + 255) & ~(size_t)255;
        GK_CUDA(dmalloc((void**)&P.unit_row, urow + (size_t)P.slots * P.carry_bytes));
        P.carries = (char*)P.unit_row + urow;
        k_unit_rows<<<grid_for(P.units + 1), 256, 0, s>>>(
            m, P.row_end ? P.row_end : A->row_ptr + 1, P.units, P.unit_row);
        GK_CUDA(cudaGetLastError());
    }
    return GK_OK;
}

// Validates a CSR handle's arrays, computes max/mean row length and plans.
// cols_valid: the columns have been checked.
static gk_status finish_csr(gk_matrix A, cudaStream_t s, bool cols_valid = false) {
    GK_TRY(ensure_words(A));
    unsigned int* derr = reinterpret_cast<unsigned int*>(A->words + 8);
    int32_t* dmax = reinterpret_cast<int32_t*>(derr + 1);
    GK_CUDA(cudaMemsetAsync(derr, 0, 16, s));
    if (A->n > 0)
        k_validate_rowptr<<<grid_for(A->n), 256, 0, s>>>(A->n, A->nnz, A->row_ptr, derr, dmax,
                                                         dmax + 1);
    if (A->nnz > 0 && !cols_valid)
        k_validate_cols<<<grid_for(A->nnz), 256, 0, s>>>(A->nnz, A->ncols, A->col, derr);
    GK_CUDA(cudaGetLastError());
    unsigned int h[3] = {0, 0, 0};
    GK_CUDA(cudaMemcpyAsync(h, derr, 12, cudaMemcpyDeviceToHost, s));
    GK_CUDA(cudaStreamSynchronize(s));
    if (h[0]) return GK_ERR_INVALID;
    A->max_row = (int32_t)h[1];
    A->empty_rows_known = (int32_t)h[2];
    A->mean_row = A->n ? (double)A->nnz / A->n : 0.0;
    GK_TRY(build_csr_plan(A, s));
    GK_CUDA(cudaStreamSynchronize(s));
    return GK_OK;
}

static gk_status copy_in(void* dst, const void* src, size_t bytes, gk_memory mem, cudaStream_t s) {
    if (bytes == 0) return GK_OK;
    if (!src) return GK_ERR_INVALID;
    GK_CUDA(cudaMemcpyAsync(dst, src, bytes,
                            mem == GK_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice,
                            s));
    return GK_OK;
}

// Whether kernels of the current device can read an array of the caller's
// where it lies: its own memory (or managed), on the element's alignment.  A
// copy takes any other device-accessible address.
static bool readable_in_place(const void* p, size_t element) {
    cudaPointerAttributes at;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return (at.type == cudaMemoryTypeManaged || (at.type == cudaMemoryTypeDevice && at.device == dev)) &&
           reinterpret_cast<uintptr_t>(p) % element == 0;
}

}  // namespace gk

using namespace gk;

extern "C" {

const char* gk_status_string(gk_status s) {
    switch (s) {
        case GK_OK: return "ok";
        case GK_NOT_CONVERGED: return "not converged: iteration cap reached";
        case GK_BREAKDOWN: return "breakdown of the Krylov recurrence";
        case GK_ERR_INVALID: return "invalid argument or malformed matrix";
        case GK_ERR_OOM: return "device memory allocation failed";
        case GK_ERR_CUDA: return "CUDA runtime error";
        case GK_ERR_TIMEOUT: return "device-side wait timed out";
        case GK_ERR_ZERO_DIAG: return "zero or missing diagonal entry (Jacobi)";
        case GK_ERR_NAN: return "NaN or Inf in a residual norm";
        case GK_ERR_UNSUPPORTED: return "unsupported combination";
    }
    return "unknown status";
}

int32_t gk_version(void) { return GK_VERSION; }

gk_status gk_matrix_create_csr(int32_t n, int32_t ncols, int64_t nnz, const int32_t* row_ptr,
                               const int32_t* col_idx, const void* values, gk_dtype dtype,
                               gk_memory mem, void* stream, gk_matrix* out) {
    if (!out) return GK_ERR_INVALID;
    *out = nullptr;
    if (n < 0 || ncols < 0 || nnz < 0 || nnz > INT32_MAX || !valid_dtype(dtype) || !row_ptr ||
        (mem != GK_MEM_HOST && mem != GK_MEM_DEVICE))
        return GK_ERR_INVALID;
    if (nnz > 0 && (!col_idx || !values)) return GK_ERR_INVALID;
    cudaStream_t s = (cudaStream_t)stream;
    gk_matrix A = new_handle();
    if (!A) return GK_ERR_OOM;
    A->n = n;
    A->ncols = ncols;
    A->nnz = nnz;
    A->fmt = GK_CSR;
    A->dtype = dtype;
    gk_status st = GK_OK;
    auto fail = [&](gk_status e) {
        destroy_handle(A);
        return e;
    };
    if ((st = alloc_csr(A)) != GK_OK) return fail(st);
    if ((st = copy_in(A->row_ptr, row_ptr, sizeof(int32_t) * ((size_t)n + 1), mem, s)) != GK_OK ||
        (st = copy_in(A->col, col_idx, sizeof(int32_t) * (size_t)nnz, mem, s)) != GK_OK ||
        (st = copy_in(A->val, values, value_bytes(dtype) * (size_t)nnz, mem, s)) != GK_OK)
        return fail(st);
    if ((st = finish_csr(A, s)) != GK_OK) return fail(st);
    *out = A;
    return GK_OK;
}

gk_status gk_matrix_create_coo(int32_t n, int32_t ncols, int64_t nnz, const int32_t* row,
                               const int32_t* col, const void* values, gk_dtype dtype,
                               gk_memory mem, void* stream, gk_matrix* out) {
    if (!out) return GK_ERR_INVALID;
    *out = nullptr;
    if (n < 0 || ncols < 0 || nnz < 0 || nnz > INT32_MAX || !valid_dtype(dtype) ||
        (mem != GK_MEM_HOST && mem != GK_MEM_DEVICE))
        return GK_ERR_INVALID;
    if (nnz > 0 && (!row || !col || !values)) return GK_ERR_INVALID;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t vb = value_bytes(dtype);
    const size_t nz1 = (size_t)std::max<int64_t>(nnz, 1), n1 = (size_t)n + 1;
    const int64_t nblk = std::max<int64_t>(1, (nnz + SCAN_TILE - 1) / SCAN_TILE);
    // one scratch allocation (an allocation and its free cost more than most
    // of the kernels); triplets on the device are read in place where they
    // can be
    size_t at = 0;
    auto part = [&](size_t bytes) {
        const size_t o = at;
        at += (bytes + 255) & ~(size_t)255;
        return o;
    };
    auto staged = [&](const void* p, size_t element) {
        return nnz > 0 && (mem == GK_MEM_HOST || !readable_in_place(p, element));
    };
    const bool copy_row = staged(row, 4), copy_col = staged(col, 4), copy_val = staged(values, vb);
    const size_t o_keys = part(8 * nz1), o_rank = part(4 * nz1), o_first = part(nz1);
    const size_t o_cnt = part(4 * n1), o_start = part(4 * n1), o_list = part(4 * n1);
    const size_t o_bsum = part(8 * (size_t)std::max(nblk + 1, n / (int64_t)SCAN_TILE + 1)), o_info = part(256);
    const size_t o_row = part(copy_row ? 4 * nz1 : 0), o_col = part(copy_col ? 4 * nz1 : 0);
    const size_t o_val = part(copy_val ? vb * nz1 : 0);
    TmpBuf scratch, longs;
    if (scratch.ensure(at)) return GK_ERR_OOM;
    char* base = static_cast<char*>(scratch.ptr);
    gk_matrix A = nullptr;
    auto fail = [&](gk_status e) {
        destroy_handle(A);
        return e;
    };
    gk_status st;
    const int32_t *drow = row, *dcol = col;
    const void* dval = values;
    if (copy_row) {
        if ((st = copy_in(base + o_row, row, 4 * (size_t)nnz, mem, s)) != GK_OK) return fail(st);
        drow = (const int32_t*)(base + o_row);
    }
    if (copy_col) {
        if ((st = copy_in(base + o_col, col, 4 * (size_t)nnz, mem, s)) != GK_OK) return fail(st);
        dcol = (const int32_t*)(base + o_col);
    }
    if (copy_val) {
        if ((st = copy_in(base + o_val, values, vb * (size_t)nnz, mem, s)) != GK_OK) return fail(st);
        dval = base + o_val;
    }
    uint64_t* dkeys = (uint64_t*)(base + o_keys);
    int32_t* drank = (int32_t*)(base + o_rank);  // then: heads before every entry
    unsigned char* dfirst = (unsigned char*)(base + o_first);
    int32_t* dcnt = (int32_t*)(base + o_cnt);
    int32_t* dstart = (int32_t*)(base + o_start);
    int32_t* dlist = (int32_t*)(base + o_list);
    int64_t* dbsum = (int64_t*)(base + o_bsum);
    // info words: the class sizes and the longest row, the error flags, the
    // lists' cursors
    int32_t* dinfo = (int32_t*)(base + o_info);
    unsigned int* derr = (unsigned int*)(dinfo + 16);
    int32_t* dcursor = dinfo + 32;
    if (cudaMemsetAsync(dinfo, 0, 256, s) || cudaMemsetAsync(dcnt, 0, 4 * n1, s) ||
        cudaMemsetAsync(dfirst, 0, nz1, s))
        return fail(GK_ERR_CUDA);
    if (nnz > 0)
        k_coo_count<<<grid_for(nnz), 256, 0, s>>>(nnz, n, ncols, drow, dcol, dcnt, drank, derr);
    if (n > 0) k_class_sizes<<<std::min(grid_for(n), (unsigned)num_sms() * 2), 256, 0, s>>>(n, dcnt, dinfo);
    if ((st = scan_exclusive_in<int32_t, int32_t>(dcnt, dstart, n, dbsum, s)) != GK_OK) return fail(st);
    int32_t info[17] = {0};
    if (cudaMemcpyAsync(info, dinfo, sizeof(info), cudaMemcpyDeviceToHost, s) ||
        cudaStreamSynchronize(s))
        return fail(GK_ERR_CUDA);
    if (info[16]) return fail(GK_ERR_INVALID);
    if (nnz > 0)
        k_coo_scatter<<<grid_for(nnz), 256, 0, s>>>(nnz, drow, dcol, dstart, drank, dkeys);
    ClassOffsets off;
    int32_t listed = 0;
    for (int c = 0; c < SORT_CLASSES; ++c) {
        off.o[c] = listed;
        listed += info[c];
    }
    if (listed > 0) {
        k_class_lists<<<(unsigned)(((int64_t)n + 255) / 256), 256, 0, s>>>(n, dcnt, off, dcursor, dlist);
        auto groups = [&](int c, int lanes) { return grid_for((int64_t)info[c] * lanes); };
        auto l = [&](int c) { return dlist + off.o[c]; };
        if (info[0]) k_sort_rows_sub<2><<<groups(0, 2), 256, 0, s>>>(info[0], l(0), dstart, dkeys);
        if (info[1]) k_sort_rows_sub<4><<<groups(1, 4), 256, 0, s>>>(info[1], l(1), dstart, dkeys);
        if (info[2]) k_sort_rows_sub<8><<<groups(2, 8), 256, 0, s>>>(info[2], l(2), dstart, dkeys);
        if (info[3]) k_sort_rows_sub<16><<<groups(3, 16), 256, 0, s>>>(info[3], l(3), dstart, dkeys);
        if (info[4]) k_sort_rows_sub<32><<<groups(4, 32), 256, 0, s>>>(info[4], l(4), dstart, dkeys);
        auto warps = [&](int c) { return (unsigned)std::min<int64_t>(((int64_t)info[c] + 3) / 4, (int64_t)num_sms() * 16); };
        if (info[5]) k_sort_rows_warp<2><<<warps(5), 128, 0, s>>>(info[5], l(5), dstart, dkeys);
        if (info[6]) k_sort_rows_warp<4><<<warps(6), 128, 0, s>>>(info[6], l(6), dstart, dkeys);
        if (info[7]) k_sort_rows_warp<8><<<warps(7), 128, 0, s>>>(info[7], l(7), dstart, dkeys);
        if (info[8]) k_sort_rows_warp<16><<<warps(8), 128, 0, s>>>(info[8], l(8), dstart, dkeys);
        const int32_t longest = info[SORT_CLASSES];
        if (info[9]) {
            cudaFuncSetAttribute(k_sort_rows_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 SORT_BLOCK_MAX * 8);
            int P = 1024;
            while (P < std::min(longest, SORT_BLOCK_MAX)) P <<= 1;
            k_sort_rows_block<<<(unsigned)std::min<int64_t>(info[9], (int64_t)num_sms() * 6), 256,
                                (size_t)P * 8, s>>>(info[9], l(9), dstart, dkeys);
        }
        if (info[10]) {
            int64_t Q = 1;
            while (Q < longest) Q <<= 1;
            const int nb = std::min(info[10], 4);
            if (longs.ensure((size_t)nb * Q * 8)) return fail(GK_ERR_OOM);
            k_sort_rows_global<<<nb, 1024, 0, s>>>(info[10], l(10), dstart, dkeys,
                                                   (uint64_t*)longs.ptr, Q);
        }
    }
    // heads: the first entry of every (row, col)
    int64_t nnz_out = 0;
    if (nnz > 0) {
        k_row_firsts<<<grid_for(n), 256, 0, s>>>(n, dstart, dfirst);
        k_head_counts<<<(unsigned)nblk, SCAN_THREADS, 0, s>>>(nnz, dkeys, dfirst, dbsum);
        if (cudaMemsetAsync(dbsum + nblk, 0, 8, s)) return fail(GK_ERR_CUDA);
        k_scan_blocksums<<<1, SCAN_THREADS, 0, s>>>(dbsum, nblk + 1);
        if (cudaMemcpyAsync(&nnz_out, dbsum + nblk, 8, cudaMemcpyDeviceToHost, s) ||
            cudaStreamSynchronize(s))
            return fail(GK_ERR_CUDA);
    }
    A = new_handle();
    if (!A) return fail(GK_ERR_OOM);
    A->n = n;
    A->ncols = ncols;
    A->nnz = nnz_out;
    A->fmt = GK_CSR;
    A->dtype = dtype;
    if ((st = alloc_csr(A)) != GK_OK) return fail(st);
    if (nnz > 0) {
        st = dispatch_dtype(dtype, [&](auto tp) -> gk_status {
            using V = typename decltype(tp)::V;
            using Acc = typename AccOf<V>::type;
            k_merge_heads<V, V, Acc><<<(unsigned)nblk, SCAN_THREADS, 0, s>>>(
                nnz, dkeys, dfirst, dbsum, (const V*)dval, drank, A->col, (V*)A->val);
            return GK_OK;
        });
        if (st != GK_OK) return fail(st);
        k_row_ptr<<<grid_for((int64_t)n + 1), 256, 0, s>>>(n, nnz, dstart, drank, dbsum + nblk,
                                                           A->row_ptr);
    } else if (cudaMemsetAsync(A->row_ptr, 0, 4 * n1, s)) {
        return fail(GK_ERR_CUDA);
    }
    if (cudaGetLastError()) return fail(GK_ERR_CUDA);
    if ((st = finish_csr(A, s, true)) != GK_OK) return fail(st);
    *out = A;
    return GK_OK;
}

gk_status gk_matrix_convert(gk_matrix A, gk_format fmt, gk_dtype dtype, int32_t slice_size,
                            int32_t stride_factor, void* stream, gk_matrix* out) {
    if (!A || !out || !valid_dtype(dtype)) return GK_ERR_INVALID;
    if (fmt != GK_CSR && fmt != GK_ELL && fmt != GK_SELLP && fmt != GK_COO) return GK_ERR_INVALID;
    *out = nullptr;
    const bool to_coo = fmt == GK_COO;
    if (to_coo) fmt = GK_CSR;  // the COO handle is a CSR handle plus the row of every entry
    cudaStream_t s = (cudaStream_t)stream;
    const int32_t S = slice_size ? slice_size : 32;
    const int32_t f = stride_factor ? stride_factor : 1;
    if (fmt == GK_SELLP && (S < 1 || S > 1024 || f < 1)) return GK_ERR_INVALID;
    // Step 1: a CSR source in the source dtype (A itself, or rebuilt from padding).
    gk_matrix C = A;
    gk_matrix tmpC = nullptr;
    auto fail = [&](gk_status e) {
        destroy_handle(tmpC);
        return e;
    };
    if (A->fmt != GK_CSR) {
        tmpC = new_handle();
        if (!tmpC) return GK_ERR_OOM;
        tmpC->n = A->n;
        tmpC->ncols = A->ncols;
        tmpC->nnz = A->nnz;
        tmpC->dtype = A->dtype;
        DevBuf cnt, tmp;
        if (cnt.ensure(4 * ((size_t)A->n + 1)) || dmalloc_t(&tmpC->row_ptr, (size_t)A->n + 1) ||
            dmalloc_t(&tmpC->col, (size_t)std::max<int64_t>(A->nnz, 1)) ||
            dmalloc(&tmpC->val, value_bytes(A->dtype) * (size_t)std::max<int64_t>(A->nnz, 1)))
            return fail(GK_ERR_OOM);
        if (A->n > 0)
            k_padded_row_counts<<<grid_for(A->n), 256, 0, s>>>(A->n, A->fmt, A->stride, A->K, A->S,
                                                               A->slice_len, A->slice_set, A->col,
                                                               (int32_t*)cnt.ptr);
        gk_status st = scan_exclusive<int32_t, int32_t>((int32_t*)cnt.ptr, tmpC->row_ptr, A->n, tmp, s);
        if (st != GK_OK) return fail(st);
        if (A->n > 0) {
            st = dispatch_dtype(A->dtype, [&](auto tp) -> gk_status {
                using V = typename decltype(tp)::V;
                k_padded_to_csr<V, V><<<grid_for(A->n), 256, 0, s>>>(
                    A->n, A->fmt, A->stride, A->K, A->S, A->slice_len, A->slice_set, A->col,
                    (const V*)A->val, tmpC->row_ptr, tmpC->col, (V*)tmpC->val);
                return GK_OK;
            });
            if (st != GK_OK) return fail(st);
        }
        if (cudaStreamSynchronize(s)) return fail(GK_ERR_CUDA);
        cnt.release();
        tmp.release();
        tmpC->max_row = A->max_row;
        C = tmpC;
    }
    gk_matrix B = new_handle();
    if (!B) return fail(GK_ERR_OOM);
    auto failB = [&](gk_status e) {
        destroy_handle(B);
        return fail(e);
    };
    B->n = A->n;
    B->ncols = A->ncols;
    B->nnz = A->nnz;
    B->fmt = fmt;
    B->dtype = dtype;
    B->max_row = A->max_row;
    B->empty_rows_known = A->empty_rows_known;
    B->mean_row = A->n ? (double)A->nnz / A->n : 0.0;
    const int64_t n = A->n;
    gk_status st = GK_OK;
    auto run = [&](auto src_tp, auto dst_tp) -> gk_status {
        using VI = typename decltype(src_tp)::V;
        using VO = typename decltype(dst_tp)::V;
        if (fmt == GK_CSR) {
            B->stored = C->nnz;
            GK_CUDA(dmalloc_t(&B->row_ptr, (size_t)n + 1));
            GK_CUDA(dmalloc_t(&B->col, (size_t)std::max<int64_t>(C->nnz, 1)));
            GK_CUDA(dmalloc(&B->val, sizeof(VO) * (size_t)std::max<int64_t>(C->nnz, 1)));
            GK_CUDA(cudaMemcpyAsync(B->row_ptr, C->row_ptr, 4 * ((size_t)n + 1), cudaMemcpyDeviceToDevice, s));
            if (C->nnz) {
                GK_CUDA(cudaMemcpyAsync(B->col, C->col, 4 * (size_t)C->nnz, cudaMemcpyDeviceToDevice, s));
                k_convert_values<VI, VO><<<grid_for(C->nnz), 256, 0, s>>>(C->nnz, (const VI*)C->val,
                                                                         (VO*)B->val);
            }
        } else if (fmt == GK_ELL) {
            B->K = C->max_row;
            B->stride = ((n + 31) / 32) * 32;
            B->stored = (int64_t)B->K * B->stride;
            GK_CUDA(dmalloc_t(&B->col, (size_t)std::max<int64_t>(B->stored, 1)));
            GK_CUDA(dmalloc(&B->val, sizeof(VO) * (size_t)std::max<int64_t>(B->stored, 1)));
            if (B->stored)
                k_csr_to_ell<VI, VO><<<grid_for(B->stride), 256, 0, s>>>(
                    (int32_t)n, B->stride, B->K, C->row_ptr, C->col, (const VI*)C->val, B->col,
                    (VO*)B->val);
        } else {
            B->S = S;
            B->f = f;
            B->nslices = (int32_t)((n + S - 1) / S);
            GK_CUDA(dmalloc_t(&B->slice_len, (size_t)std::max(B->nslices, 1)));
            GK_CUDA(dmalloc_t(&B->slice_set, (size_t)B->nslices + 1));
            if (B->nslices)
                k_slice_lengths<<<grid_for(B->nslices), 256, 0, s>>>((int32_t)n, S, f, B->nslices,
                                                                    C->row_ptr, B->slice_len);
            DevBuf tmp;
            GK_TRY(scan_exclusive<int32_t, int64_t>(B->slice_len, B->slice_set, B->nslices, tmp, s));
            int64_t total = 0;
            GK_CUDA(cudaMemcpyAsync(&total, B->slice_set + B->nslices, 8, cudaMemcpyDeviceToHost, s));
            GK_CUDA(cudaStreamSynchronize(s));
            tmp.release();
            B->stored = total * S;
            GK_CUDA(dmalloc_t(&B->col, (size_t)std::max<int64_t>(B->stored, 1)));
            GK_CUDA(dmalloc(&B->val, sizeof(VO) * (size_t)std::max<int64_t>(B->stored, 1)));
            if (B->nslices)
                k_csr_to_sellp<VI, VO><<<grid_for((int64_t)B->nslices * S), 256, 0, s>>>(
                    (int32_t)n, S, B->nslices, C->row_ptr, C->col, (const VI*)C->val,
                    B->slice_len, B->slice_set, B->col, (VO*)B->val);
        }
        GK_CUDA(cudaGetLastError());
        return GK_OK;
    };
    st = dispatch_dtype(C->dtype, [&](auto src) {
        return dispatch_dtype(dtype, [&](auto dst) { return run(src, dst); });
    });
    if (st != GK_OK) return failB(st);
    if (fmt == GK_CSR && (st = build_csr_plan(B, s)) != GK_OK) return failB(st);
    if (to_coo && (st = build_coo_view(B, s)) != GK_OK) return failB(st);
    if (cudaStreamSynchronize(s)) return failB(GK_ERR_CUDA);
    destroy_handle(tmpC);
    *out = B;
    return GK_OK;
}

gk_status gk_matrix_describe(gk_matrix A, gk_matrix_desc* d) {
    if (!A || !d) return GK_ERR_INVALID;
    std::memset(d, 0, sizeof(*d));
    d->n = A->n;
    d->ncols = A->ncols;
    d->nnz = A->nnz;
    d->format = A->coo ? GK_COO : A->fmt;
    d->dtype = A->dtype;
    d->max_row = A->max_row;
    d->ell_width = A->K;
    d->ell_stride = A->stride;
    d->slice_size = A->S;
    d->stride_factor = A->f;
    d->num_slices = A->nslices;
    d->spmv_kernel = A->coo ? 5
                     : A->fmt == GK_CSR ? (A->plan.seg ? 2 : A->plan.kind == 3 ? 6 : A->plan.kind)
                     : A->fmt == GK_ELL ? 3 : 4;
    if (A->plan.err) {
        int32_t e = 0;
        if (cudaMemcpy(&e, A->plan.err, 4, cudaMemcpyDeviceToHost) == cudaSuccess && e)
            d->device_error |= 1;
    }
    // the substitution kernels' sticky error words (TriStore::sync: four
    // words per direction, the third is the error flag)
    const gk::TriStore* tri[2] = {A->ilu, A->tri};
    for (int k = 0; k < 2; ++k) {
        if (!tri[k] || tri[k]->state != 1 || !tri[k]->sync) continue;
        uint32_t w[8] = {};
        if (cudaMemcpy(w, tri[k]->sync, sizeof(w), cudaMemcpyDeviceToHost) == cudaSuccess &&
            (w[2] | w[6]))
            d->device_error |= 2 << k;
    }
    d->spmv_launches = A->coo ? (A->n_empty ? 3 : 2)
                       : (A->fmt == GK_CSR && A->plan.seg) ? (A->plan.n_empty ? 3 : 2) : 1;
    d->solve_format = A->fmt != GK_CSR ? (int32_t)A->fmt
                      : !A->solve_fmt_tuned ? -1
                      : A->solve_fmt ? (int32_t)A->solve_fmt->fmt : (int32_t)GK_CSR;
    const size_t vb = value_bytes(A->dtype);
    if (A->fmt == GK_CSR) {
        d->stored = A->nnz;
        d->device_bytes = (int64_t)(4 * ((size_t)A->n + 1) + (4 + vb) * (size_t)A->nnz);
        if (A->coo) d->device_bytes += (int64_t)(4 * (size_t)A->nnz + 4 * (size_t)A->n_empty);
    } else if (A->fmt == GK_ELL) {
        d->stored = A->stored;
        d->device_bytes = (int64_t)((4 + vb) * (size_t)A->stored);
    } else {
        d->stored = A->stored;
        d->device_bytes = (int64_t)((4 + vb) * (size_t)A->stored + 4 * (size_t)A->nslices +
                                    8 * ((size_t)A->nslices + 1));
    }
    return GK_OK;
}

gk_status gk_matrix_export(gk_matrix A, int32_t* idx_a, int64_t* sets, int32_t* col, void* values) {
    if (!A) return GK_ERR_INVALID;
    GateShared gate;
    GK_CUDA(cudaDeviceSynchronize());
    const size_t vb = value_bytes(A->dtype);
    if (A->coo) {
        if (idx_a && A->nnz) GK_CUDA(cudaMemcpy(idx_a, A->coo_row, 4 * (size_t)A->nnz, cudaMemcpyDeviceToHost));
        if (col && A->nnz) GK_CUDA(cudaMemcpy(col, A->col, 4 * (size_t)A->nnz, cudaMemcpyDeviceToHost));
        if (values && A->nnz) GK_CUDA(cudaMemcpy(values, A->val, vb * (size_t)A->nnz, cudaMemcpyDeviceToHost));
    } else if (A->fmt == GK_CSR) {
        if (idx_a) GK_CUDA(cudaMemcpy(idx_a, A->row_ptr, 4 * ((size_t)A->n + 1), cudaMemcpyDeviceToHost));
        if (col && A->nnz) GK_CUDA(cudaMemcpy(col, A->col, 4 * (size_t)A->nnz, cudaMemcpyDeviceToHost));
        if (values && A->nnz) GK_CUDA(cudaMemcpy(values, A->val, vb * (size_t)A->nnz, cudaMemcpyDeviceToHost));
    } else {
        if (A->fmt == GK_SELLP) {
            if (idx_a && A->nslices)
                GK_CUDA(cudaMemcpy(idx_a, A->slice_len, 4 * (size_t)A->nslices, cudaMemcpyDeviceToHost));
            if (sets) GK_CUDA(cudaMemcpy(sets, A->slice_set, 8 * ((size_t)A->nslices + 1), cudaMemcpyDeviceToHost));
        }
        if (col && A->stored) GK_CUDA(cudaMemcpy(col, A->col, 4 * (size_t)A->stored, cudaMemcpyDeviceToHost));
        if (values && A->stored)
            GK_CUDA(cudaMemcpy(values, A->val, vb * (size_t)A->stored, cudaMemcpyDeviceToHost));
    }
    return GK_OK;
}

gk_status gk_matrix_destroy(gk_matrix A) {
    if (!A) return GK_ERR_INVALID;
    GateShared gate;  // streams, graphs, events and memory go: no capture meanwhile
    cudaDeviceSynchronize();
    destroy_handle(A);
    return GK_OK;
}

}  // extern "C"
