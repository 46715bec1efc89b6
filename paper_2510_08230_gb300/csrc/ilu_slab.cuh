// ilu_slab.cuh - slab mode of the ILU(0) substitutions: consecutive rows stay
// on one SM, and only values that cross a slab's boundary go through L2.
//
// Dependency levels bound a substitution: 382 a triangle on a 128^3 stencil.
// The window mode takes all SMs it uses through one cluster barrier a level
// (2.1 us).  Here a block owns a slab of consecutive rows and walks its
// own levels with a block barrier each; a slab only trails the one before it
// by a hand-off through L2 (~0.7 us), paid once a slab boundary on the longest
// dependency path instead of once a level.  What is left of a level (stamps,
// cycles): the row's dependent FP64 operations 90 each, the reads of its
// values and of the next level's records 150, the stores 100, decoding 70,
// barrier and loop 170: ~800 on the 7-point stencil, ~600 in FP32.
//
// One application (GB300, us), window mode / this one: 128^3 diffusion FP64
// 1,650 / 570, FP32 1,242 / 435; 2D 1024^2 4,892 / 1,301; 200 x 200 x 20
// 1,123 / 405; 2D 64^2 337 / 191.  120 applications from six threads, 128^3:
// 36.4 ms / 20.1 (two blocks an SM; with eight polling warps only one fits
// without spills).  On the way, 128^3 FP64: the computing
// threads also copying and testing the barriers 1,110, a copying warp 753,
// addresses precomputed in the records 735, a warp that waits on their
// behalf 680, the number of terms a constant (a predicated FP64 operation
// costs as much as an executed one) 565.
//
// A block: SLAB_CT threads compute, a row each (up to SLAB_RPT); SLAB_PW
// warps fetch the values that rows of the next levels need from other slabs:
// warp p polls those of levels p, p + SLAB_PW, ... into a ring of SLAB_E
// levels in shared memory, so a level's polls overlap the ones before it.
// A value is its own ready signal, as in the chunked kernel (a signalling
// NaN marks an unsolved slot); values are handed over in level order (the
// rows of a level side by side), beside the caller's vector.  Values the
// slab's own rows need stay in a ring of the last WIN_MAXD + 1 levels.
// Two threads bulk-copy records and level-ordered inputs up to nb levels
// ahead, and one warp waits for copies and fetched values on the computing
// warps' behalf and joins their barrier, so that they test nothing.  Every
// row's subtractions keep the substitution order: the result is bit-identical
// to the other modes.
//
// No wait can be circular: a slab only waits on slabs of rows before it (U:
// after it), and blocks claim slabs in that order from a counter.  Every wait
// takes the caller's budget: for the block's own copies, as in the window
// mode, and for other slabs' values, as in the chunked kernels (the last slab
// starts only when the wavefront arrives, so a budget below a triangle's time
// runs out there).  When one runs out, all later ones give up at once and the
// launch ends with wrong values and the error word.
#pragma once

namespace gk {

constexpr int SLAB_CT = 256;    // computing threads
constexpr int SLAB_PW = 4;      // polling warps
constexpr int SLAB_SW = 2;      // copying warps
constexpr int SLAB_NT = SLAB_CT + 32 * (SLAB_PW + SLAB_SW + 1);
constexpr int SLAB_RPT = 3;     // rows of a level per thread at most
constexpr int SLAB_CAP = SLAB_RPT * SLAB_CT;
constexpr int SLAB_E = 16;      // levels of fetched values kept
constexpr int SLAB_NB = 8;      // levels of records in flight at most (always even)
constexpr int SLAB_SMEM = 226 * 1024;  // dynamic shared memory at most
constexpr int SLAB_SLOTS = WIN_MAXD + 1;
// WinRec::co of this mode: the index of the term's value in the block's
// values: first SLAB_ZERO zeros (terms past the row's: subtracting 0 * 0
// changes nothing), then SLAB_E levels of fetched values, then the ring.
// Level e of the slab (from 0) keeps its fetched and own values at:
constexpr int SLAB_ZERO = 2;
__host__ __device__ inline int slab_ext_at(int e, int ecap) { return SLAB_ZERO + e % SLAB_E * ecap; }
__host__ __device__ inline int slab_ring_at(int e, int cap, int ecap) {
    return SLAB_ZERO + SLAB_E * ecap + e % SLAB_SLOTS * cap;
}
__host__ __device__ inline int slab_values(int cap, int ecap) {
    return SLAB_ZERO + SLAB_E * ecap + SLAB_SLOTS * cap;
}
static_assert(SLAB_E >= SLAB_PW, "every polling warp has a level to fetch into");

// bytes of dynamic shared memory (cap: a multiple of 4, so that every buffer
// starts on 16 bytes)
template <typename T>
__host__ __device__ inline size_t slab_smem(int cap, int ecap, int nb) {
    constexpr int AL = (int)(16 / sizeof(T));
    return (size_t)nb * ((size_t)cap * sizeof(WinRec<T>) + (size_t)(cap + 2 * AL) * sizeof(T) +
                         (size_t)(cap + 8) * 4) +
           (size_t)slab_values(cap, ecap) * sizeof(T);
}

__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void lds(double& v, uint32_t a) {
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a));
}
__device__ __forceinline__ void lds(float& v, uint32_t a) {
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
}

// RPT: rows of a level per thread (1 or SLAB_RPT, by the widest bucket)
template <typename T, bool UP, int RPT, class Out, class Skip, class Err>
__global__ void __launch_bounds__(SLAB_NT, RPT == 1 ? 2 : 1)
k_ilu_trsv_slab(IluDev<T> f, Out out, Skip sk, Err on_err) {
    if (sk.skip()) return;
    constexpr int AL = (int)(16 / sizeof(T));
    extern __shared__ __align__(128) unsigned char ssm[];
    __shared__ uint64_t full_rec[SLAB_NB], full_ext[SLAB_E];
    __shared__ int s_claim;
    __shared__ volatile int s_dead;  // a wait of this block ran out
    __shared__ volatile int s_done;  // levels of the slab that have ended
    const SlabDir& D = f.sd[UP ? 1 : 0];
    const int cap = D.cap, ecap = D.ecap, nb = D.nb;
    WinRec<T>* recs = reinterpret_cast<WinRec<T>*>(ssm);
    T* ins = reinterpret_cast<T*>(recs + (size_t)nb * cap);
    int32_t* rws = reinterpret_cast<int32_t*>(ins + (size_t)nb * (cap + 2 * AL));
    T* vals = reinterpret_cast<T*>(rws + (size_t)nb * (cap + 8));
    TrsvSync* sy = f.sy + (UP ? 1 : 0);
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) {
        s_claim = (int)atomicAdd(&sy->ctr, 1u);
        s_dead = 0;
        s_done = -1;
        for (int i = 0; i < SLAB_ZERO; ++i) vals[i] = T(0);
        for (int i = 0; i < nb; ++i) mbar_init(smem_addr(full_rec + i), 1);
        for (int i = 0; i < SLAB_E; ++i) mbar_init(smem_addr(full_ext + i), 1);
        fence_mbar_init();
    }
    __syncthreads();
    const int slab = UP ? D.nslab - 1 - s_claim : s_claim;
    const int32_t lo = D.range[2 * slab], hi = D.range[2 * slab + 1];
    T* hand = f.shand;
    const int32_t* start = D.start + (size_t)slab * D.nlev;
    int32_t staged = 0;  // copying threads: one past the last level copied or under way
    auto give_up = [&]() {
        s_dead = 1;
        atomicExch(&sy->err, 1u);
    };
    // a wait on other warps of this block, which give up first: they wait at
    // most the budget for a value
    auto wait_block = [&](auto ready) {
        uint64_t t0 = 0;
        while (!s_dead) {
            for (int k = 0; k < 64; ++k)
                if (ready()) return;
            const uint64_t t = globaltimer_ns();
            if (t0 == 0) t0 = t;
            if ((t - t0) / 2 > f.wait_ns) give_up();
        }
    };
    // until `want` levels have ended
    auto wait_done = [&](int32_t want) {
        wait_block([&] {
            if (s_done >= want) return true;
            __nanosleep(100);  // leaves the issue slots to the computing warps
            return false;
        });
        __threadfence_block();
    };
    // ends a level: the computing warps and the one that waits for them
    auto barrier = [] { asm volatile("bar.sync 1, %0;" ::"n"(SLAB_CT + 32) : "memory"); };

    if (tid < SLAB_CT) {
        // level L's rows of this thread, and what the next level's need
        T v[RPT][WIN_MAXT], rd[RPT], in[RPT];
        uint32_t ad[RPT][WIN_MAXT];  // shared-memory addresses of the terms' values
        int32_t at[RPT], row[RPT];   // position in level order (-1: none), row
        const uint32_t vals_a = smem_addr(vals);
        const int w0 = tid & ~31;
        int buf = 0;  // of the level read last
        struct Raw {
            WinRec<T> W;
            T in;
            int32_t row, at;
        } Y[RPT];
        // bucket [a, b) from its buffer.  It has landed before the last barrier
        // unless a wait ran out: then no record is used.
        auto read = [&](int32_t a, int32_t b) {
            const bool dead = s_dead != 0;
            const WinRec<T>* sr = recs + (size_t)buf * cap;
            const T* si = ins + (size_t)buf * (cap + 2 * AL) + (a & (AL - 1));
            const int32_t* sw = rws + (size_t)buf * (cap + 8) + (a & 3);
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const int32_t q = tid + r * SLAB_CT;
                const bool has = a + q < b;
                const int32_t i = has ? q : 0;
                Y[r].W = sr[i];
                Y[r].in = si[i];
                Y[r].row = sw[i];
                Y[r].at = has && !dead ? a + q : -1;
            }
        };
        auto decode = [&]() {
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                at[r] = Y[r].at;
                row[r] = Y[r].row;
                rd[r] = Y[r].W.rd;
                in[r] = Y[r].in;
#pragma unroll
                for (int t = 0; t < WIN_MAXT; ++t) {
                    v[r][t] = Y[r].W.v[t];
                    ad[r][t] = vals_a + (at[r] >= 0 ? (uint32_t)(uint16_t)Y[r].W.co[t] : 0u) * (uint32_t)sizeof(T);
                }
            }
        };
        int32_t a1 = start[lo], b1 = start[lo + 1];  // the bucket read last
        int32_t ahead = lo < hi ? start[lo + 2] : 0;
        barrier();
        read(a1, b1);
        decode();
        barrier();
        T* dst = out.dst();
        int slot = 0;
        T* const ring = vals + slab_ring_at(0, cap, ecap);
        // MT: terms of a row at most (a predicated FP64 operation costs as much
        // as an executed one)
        auto levels = [&](auto terms) {
            constexpr int MT = decltype(terms)::value;
            for (int32_t L = lo;; ++L) {
                const int32_t a0 = a1, b0 = b1;
                a1 = b0;
                b1 = L < hi ? ahead : b0;
                if (L + 1 < hi) ahead = start[L + 3];
                if (++buf == nb) buf = 0;
                // a warp without rows in this level or the next has nothing to do
                const bool some0 = a0 + w0 < b0, some1 = a1 + w0 < b1;
                T y[RPT];
                int32_t cat[RPT], crow[RPT];
#pragma unroll
                for (int r = 0; r < RPT; ++r) cat[r] = -1;
                if (some0 || some1) {
                    T z[RPT][WIN_MAXT];
                    if (some0) {
#pragma unroll
                        for (int r = 0; r < RPT; ++r)
#pragma unroll
                            for (int t = 0; t < MT; ++t) lds(z[r][t], ad[r][t]);
                    }
                    read(a1, b1);
                    if (some0) {
#pragma unroll
                        for (int r = 0; r < RPT; ++r) {
                            if (r > 0 && a0 + w0 + r * SLAB_CT >= b0) break;
                            T acc = in[r];
#pragma unroll
                            for (int t = 0; t < MT; ++t) acc = sub_mul(acc, v[r][t], z[r][t]);
                            if (UP) acc = mul_rn(acc, f.udiag ? rd[r] : T(1));
                            else if (f.ldiag) acc = mul_rn(acc, rd[r]);
                            y[r] = acc;
                            cat[r] = at[r];
                            crow[r] = row[r];
                            if (cat[r] >= 0) {
                                ring[slot * cap + tid + r * SLAB_CT] = acc;
                                st_relaxed_v(hand + cat[r], acc);
                            }
                        }
                    }
                    decode();
                }
                if (++slot == SLAB_SLOTS) slot = 0;
                barrier();
#pragma unroll
                for (int r = 0; r < RPT; ++r)
                    if (cat[r] >= 0) {
                        dst[crow[r]] = y[r];
                        out.extra(crow[r], y[r]);
                    }
                if (L == hi) break;
            }
        };
        if (D.terms <= 2) levels(std::integral_constant<int, 2>{});
        else if (D.terms == 3) levels(std::integral_constant<int, 3>{});
        else levels(std::integral_constant<int, WIN_MAXT>{});
    } else if (tid >= SLAB_CT + 32 * (SLAB_PW + SLAB_SW)) {
        // The barrier that ends level e: before it, what level e + 1 uses is
        // there (its fetched values, the records of the level after it); after
        // it every warp has read level e + 1's records and e's fetched values.
        auto landed = [&](uint32_t bar, uint32_t parity) {
            if (!s_dead && !win_wait(bar, parity, f.wait_ns)) give_up();
        };
        landed(smem_addr(full_rec), 0u);
        barrier();
        int buf = 1 % nb;  // of level e + 2
        uint32_t rph = 0;
        for (int32_t e = -1; lo + e <= hi; ++e) {
            const uint32_t rb = smem_addr(full_rec + buf);
            const uint32_t eb = smem_addr(full_ext + (e + 1) % SLAB_E), eph = (uint32_t)((e + 1) / SLAB_E) & 1u;
            const bool more = lo + e + 1 <= hi, more2 = lo + e + 2 <= hi;
            const bool r_there = mbar_test(rb, rph), e_there = mbar_test(eb, eph);
            if (more2 && !r_there) landed(rb, rph);
            if (more && !e_there) wait_block([&] { return mbar_test(eb, eph); });
            __syncwarp();
            barrier();
            if (lane == 0) {
                __threadfence_block();
                s_done = e + 1;
            }
            if (++buf == nb) {
                buf = 0;
                rph ^= 1u;
            }
        }
    } else if (tid >= SLAB_CT + 32 * SLAB_PW) {
        if (lane == 0) {
            const int k = (tid - SLAB_CT) / 32 - SLAB_PW;
            for (int32_t e = k; lo + e <= hi; e += SLAB_SW) {
                const int32_t a = start[lo + e], b = start[lo + e + 1];
                const int buf = e % nb;
                const uint32_t bar = smem_addr(full_rec + buf);
                const int32_t ia = a & ~(AL - 1), ib = (b + AL - 1) & ~(AL - 1);
                const int32_t wa = a & ~3, wb = (b + 3) & ~3;
                const uint32_t rn = (uint32_t)(b - a) * (uint32_t)sizeof(WinRec<T>);
                const uint32_t in = (uint32_t)(ib - ia) * (uint32_t)sizeof(T);
                const uint32_t wn = (uint32_t)(wb - wa) * 4u;
                // level e - nb, whose buffer this is, has been read
                if (e >= nb) wait_done(e - nb);
                if (s_dead) break;
                fence_proxy_async_smem();
                mbar_arrive_expect_tx(bar, b > a ? rn + in + wn : 0u);
                if (b > a) {
                    bulk_g2s(smem_addr(recs + (size_t)buf * cap),
                             static_cast<const WinRec<T>*>(D.rec) + a, rn, bar);
                    bulk_g2s(smem_addr(ins + (size_t)buf * (cap + 2 * AL)), f.sperm + ia, in, bar);
                    bulk_g2s(smem_addr(rws + (size_t)buf * (cap + 8)), D.rows + wa, wn, bar);
                }
                staged = e + 1;
            }
        }
    } else {
        constexpr int PU = 4;  // values in flight a lane
        const int32_t* estart = D.estart + (size_t)slab * D.nlev;
        for (int32_t e = (tid - SLAB_CT) >> 5; lo + e <= hi; e += SLAB_PW) {
            const int es = e % SLAB_E;
            const int32_t k0 = estart[lo + e], ne = estart[lo + e + 1] - k0;
            if (e >= SLAB_E) wait_done(e - SLAB_E + 1);  // the slot's last values are used
            for (int32_t base = lane; base < ne; base += 32 * PU) {
                const T* p[PU];
                T v[PU];
                unsigned open = 0;
#pragma unroll
                for (int u = 0; u < PU; ++u)
                    if (base + 32 * u < ne) {
                        p[u] = hand + D.epos[k0 + base + 32 * u];
                        open |= 1u << u;
                    }
                uint64_t t0 = 0;
                for (unsigned spin = 1;; ++spin) {
#pragma unroll
                    for (int u = 0; u < PU; ++u)
                        if (open >> u & 1) v[u] = ld_relaxed_v(p[u]);
#pragma unroll
                    for (int u = 0; u < PU; ++u)
                        if ((open >> u & 1) && !Sentinel<T>::is(v[u])) open &= ~(1u << u);
                    if (!open) break;
                    if (spin % 16 == 0) {
                        const uint64_t t = globaltimer_ns();
                        if (t0 == 0) t0 = t;
                        if (s_dead || ld_relaxed_u32(&sy->err) != 0u) break;
                        if (t - t0 > f.wait_ns) {
                            give_up();
                            break;
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < PU; ++u)
                    if (base + 32 * u < ne) vals[slab_ext_at(es, ecap) + base + 32 * u] = v[u];
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(full_ext + es));
        }
    }
    __syncthreads();
    // a wait ran out: the shared memory must outlive the copies in flight
    // (each copying thread waits, with the default limit, for its last one
    // into each of its buffers: nb is even)
    if (s_dead && staged > 0)
        for (int32_t e = staged - 1; e >= 0 && e > staged - 1 - nb; e -= SLAB_SW)
            mbar_wait_bounded(smem_addr(full_rec + e % nb), (uint32_t)(e / nb) & 1u);
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(&sy->exited, 1u) == gridDim.x - 1) {
            if (UP) on_err(ld_acquire_u32(&f.sy[0].err) | ld_acquire_u32(&f.sy[1].err));
            sy->ctr = 0;
            sy->exited = 0;
            __threadfence();
        }
    }
}

// The input in level order (a signalling NaN quieted, as in the other
// modes), and every hand-off slot marked unsolved.
template <typename T, class Src, class Skip>
__global__ void __launch_bounds__(256)
k_slab_prep(int32_t n, const int32_t* __restrict__ rows, Src src, T* __restrict__ perm,
            T* __restrict__ hand, Skip sk) {
    if (sk.skip()) return;
    const T* in = src.ptr();
    const T s = Sentinel<T>::value();
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
         idx += (int64_t)gridDim.x * blockDim.x) {
        perm[idx] = mul_rn(in[rows[idx]], T(1));
        hand[idx] = s;
    }
}

template <typename T, bool UP, class Src, class Out, class Skip, class Err>
static gk_status launch_slab(const IluDev<T>& f, Src src, Out out, Skip sk, Err on_err,
                             cudaStream_t s) {
    const SlabDir& D = f.sd[UP ? 1 : 0];
    auto k1 = k_ilu_trsv_slab<T, UP, 1, Out, Skip, Err>;
    auto kn = k_ilu_trsv_slab<T, UP, SLAB_RPT, Out, Skip, Err>;
    // an attribute of the functions, not a stream operation: set once
    static std::atomic<bool> attr{false};
    if (!attr.load(std::memory_order_acquire)) {
        GK_CUDA(cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, SLAB_SMEM));
        GK_CUDA(cudaFuncSetAttribute(kn, cudaFuncAttributeMaxDynamicSharedMemorySize, SLAB_SMEM));
        attr.store(true, std::memory_order_release);
    }
    const unsigned g = (unsigned)std::max<int64_t>(
        1, std::min<int64_t>(((int64_t)f.n + 1023) / 1024, (int64_t)num_sms() * 8));
    k_slab_prep<T, Src, Skip><<<g, 256, 0, s>>>(f.n, D.rows, src, f.sperm, f.shand, sk);
    (D.cap <= SLAB_CT ? k1 : kn)<<<(unsigned)D.nslab, SLAB_NT,
                                   slab_smem<T>(D.cap, D.ecap, D.nb), s>>>(f, out, sk, on_err);
    GK_CUDA(cudaGetLastError());
    return GK_OK;
}

}  // namespace gk
