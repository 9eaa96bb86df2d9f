// route.cu -- batched semantic routing of the paper's front end (Sec. 3.1):
// the score of request x against group G_i is the cosine similarity of its
// embedding with the group's centroid, the request goes to the best group
// i* = argmax_i S (lowest i on ties), or to the cache-miss branch when
// S(x, G_i*) < tau.
//
// The scores are one GEMM, E C^T, with the arg max fused into its epilogue
// (the B x N score matrix never reaches memory):
//   route_gemm_kernel: a CTA owns 128 requests (MMA M) and a contiguous range
//     of 128-group tiles.  Warp 0 streams the CTA's embedding rows, once, and
//     the centroids through a TMA ring, 128 dims a stage (a box per 64 dims,
//     128-byte swizzle); warp 1 copies the embedding rows to tensor memory as
//     they land (up to 192 columns), where every MMA reads them, and issues
//     tcgen05.mma (M = 128, N = 128, K = 16 per instruction, fp32 accumulators
//     in tensor memory, two buffers); warps 4-11 take one row and half a
//     tile's columns each per thread, scale each dot product by the
//     centroid's inverse norm and keep the running maximum and its lowest
//     index.
//     What bounds it: a tile is 24 MMAs of 64 cycles at 384 dims, and the two
//     issuing warps and the epilogue have to keep below that.  Both issuing
//     warps run their loops with all lanes and elect one to issue: a lone lane
//     beside 31 parked at the block barrier took 450 cycles for each 64 dims
//     without its MMAs (a tile 4140 cycles; loads or none made no
//     difference).  1024 requests, 16384 groups, 384 dims, both kernels in a
//     captured graph: 23.8 us so, 17.1 as it is; a further 1024 requests 14.6
//     and 8.2.
//   route_merge_kernel: one warp per request folds the CTAs' partials (score
//     first, then lower index), applies the request's own inverse norm and
//     the threshold.
//   route_norms_kernel: inverse L2 norms of the centroids (the group index
//     changes slowly, so this runs when it changes, not per batch).
#include <cudaTypedefs.h>

#include "cs_device.cuh"
#include "cs_internal.h"

namespace cs {
namespace {

constexpr int kRM = 128;                  // requests per tile (MMA M)
constexpr int kRN = 128;                  // groups per tile (MMA N)
constexpr int kKC = 64;                   // dims per box: one 128-byte swizzle row
constexpr int kBoxBytes = kRM * 128;      // 128 rows x 64 dims x 2 B
constexpr int kStageBoxes = 2;            // boxes of 128 groups a ring stage holds
constexpr int kStageBytes = kStageBoxes * kBoxBytes;
constexpr int kSlots = 7;                 // ring stages
constexpr int kEpiWarps = 8;              // two to a quarter of the rows, 64 columns of a tile each
constexpr int kRThreads = 128 + kEpiWarps * 32;   // warp 0 TMA, warp 1 MMA, warp 2 TMEM, warps 4-11 epilogue
constexpr int kRACol = 2 * kRN;           // tensor memory: two accumulators, then the request tile
constexpr int kRTmemCols = 512;
constexpr int kRTailBytes = 256 /*barriers*/ + 2 * kRN * 4 /*inverse norms*/ + kRM * 8 /*column halves*/ + 16;
constexpr int kRSmemBytes = kSlots * kStageBytes + kRTailBytes;
static_assert(kRSmemBytes <= 232448, "shared memory per block on sm_103a");
static_assert(kRACol + kMaxRouteDim / 2 <= kRTmemCols, "tensor memory");

struct RouteParams {
    int B, N, n_boxes, n_tiles, grid, seg_slots;
    long long items;              // m_tiles * n_tiles work items, split evenly over the grid
    const float* inv_norm_c;      // [N]
    float2* part;                 // [m_tiles, seg_slots, 128]: (max of dot * inv_norm_c, index as int bits)
    int* status;
};

// The CTA whose item range holds item x: ranges are [c*I/G, (c+1)*I/G).
__host__ __device__ __forceinline__ int route_owner(long long x, long long items, int grid) {
    return (int)(((x + 1) * grid + items - 1) / items) - 1;
}

__host__ __device__ constexpr uint32_t route_idesc() {
    // kind::f16: bf16 A and B (both K-major), fp32 D, M = 128, N = 128
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kRN >> 3) << 17) | ((uint32_t)(kRM >> 4) << 24);
}

__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr) {
    // 128-byte swizzle, K-major: 8-row groups 1024 bytes apart
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tc_mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, q;\n\t}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

// The whole warp spins (no suspend) on the phase; about one second at most,
// then records the timeout in the status word.  The result is the same in
// every lane, so that no lane leaves a loop while another still issues.
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, int* status) {
    if (__all_sync(0xffffffffu, mbar_test_wait(bar, parity))) return true;
    uint64_t t0 = 0;
    bool done = false;
    for (uint32_t it = 0; it < (1u << 28) && !done; ++it) {
        done = mbar_test_wait(bar, parity);
        if ((it & 1023u) == 1023u) {
            const uint64_t now = global_timer_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > 1000000000ull) break;
        }
    }
    if (!done) atomicOr(status, CS_DEVICE_WAIT_TIMEOUT);
    return __all_sync(0xffffffffu, done);
}

// 32 columns of this warp's 32 rows.
__device__ __forceinline__ void tmem_ld32(uint32_t (&r)[32], uint32_t addr) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(addr));
}

// The epilogue warps of one column half (ids 1, 2), and all of them (id 3).
__device__ __forceinline__ void epi_half_sync(int half) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + half), "n"(kEpiWarps * 16) : "memory");
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 3, %0;" ::"n"(kEpiWarps * 32) : "memory"); }

// Persistent: CTA c owns the work items [c*I/G, (c+1)*I/G) of the m-major
// sequence (request tile m, group tile t).  The request tile stays resident
// in tensor memory while t advances and is reloaded when m changes: a stage
// of its dims comes before each stage of the first group tile's.  (Read from
// shared memory, an MMA of 128 x 128 x 16 moves 8 KB of operands in the 64
// cycles it takes, all that shared memory has: 46.1 us for 4096 requests and
// 16384 groups of 384 dims, 41.7 from tensor memory; 1024 requests 17.8 and
// 17.1.  The stream of centroids is the next bound: 98 KB a tile, 1.2 us.)
__global__ void __launch_bounds__(kRThreads, 1)
route_gemm_kernel(const __grid_constant__ CUtensorMap tmap_e, const __grid_constant__ CUtensorMap tmap_c,
                  const RouteParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* tail = smem + kSlots * kStageBytes;          // after the ring: [kSlots][2 boxes][128 rows][128 B]
    uint64_t* a_free = reinterpret_cast<uint64_t*>(tail);
    uint64_t* d_full = a_free + 1;           // [2]
    uint64_t* d_free = a_free + 3;           // [2]
    uint64_t* mma_done = a_free + 5;
    uint64_t* full = a_free + 6;             // [kSlots]
    uint64_t* empty = full + kSlots;         // [kSlots]
    float* s_inv = reinterpret_cast<float*>(tail + 256);                   // [2][128]
    float2* s_half = reinterpret_cast<float2*>(tail + 256 + 2 * kRN * 4);   // [128]
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(tail + 256 + 2 * kRN * 4 + kRM * 8);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long it0 = (long long)blockIdx.x * p.items / p.grid;
    const long long it1 = (long long)(blockIdx.x + 1) * p.items / p.grid;
    const int nt = (int)(it1 - it0);
    int m = (int)(it0 / p.n_tiles), t = (int)(it0 - (long long)m * p.n_tiles);   // the current item
    const int n_kc = (p.n_boxes + kStageBoxes - 1) / kStageBoxes;               // stages a tile
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                     "n"(kRTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        tma_prefetch_desc(&tmap_e);
        tma_prefetch_desc(&tmap_c);
        mbar_init(a_free, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&d_full[i], 1);
            mbar_init(&d_free[i], kEpiWarps);
        }
        mbar_init(mma_done, 1);
        for (int i = 0; i < kSlots; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        fence_barrier_init();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *s_tmem;
    wait_prior_grid();
    allow_dependent_launch();

    if (warp == 0) {
        // ---------------------------------------------------------- TMA
        const uint32_t base = smem_u32(smem);
        int s = 0;
        uint32_t use = 0;
        long long fills = 0;
        bool ok = true, new_m = true;
        auto load = [&](const CUtensorMap* map, int kc, int row0) {
            if (use > 0 && !wait_bar(&empty[s], (use - 1) & 1, p.status)) return false;
            if (elect_one()) {
                const int k0 = kc * kStageBoxes, nb = min(kStageBoxes, p.n_boxes - k0);
                mbar_arrive_expect_tx(&full[s], (uint32_t)(nb * kBoxBytes));
                for (int k = 0; k < nb; ++k)
                    tma_load_2d(base + s * kStageBytes + k * kBoxBytes, map, &full[s], (k0 + k) * kKC, row0);
            }
            __syncwarp();
            ++fills;
            if (++s == kSlots) {
                s = 0;
                ++use;
            }
            return true;
        };
        for (int tl = 0; tl < nt && ok; ++tl) {
            for (int kc = 0; kc < n_kc && ok; ++kc) {
                if (new_m) ok = load(&tmap_e, kc, m * kRM);
                ok = ok && load(&tmap_c, kc, t * kRN);
            }
            new_m = ++t == p.n_tiles;
            if (new_m) {
                t = 0;
                ++m;
            }
        }
        // no copy in flight at exit: the last fill of every slot has landed
        for (long long f = fills > kSlots ? fills - kSlots : 0; f < fills; ++f)
            if (!mbar_wait_bounded(&full[f % kSlots], (uint32_t)(f / kSlots) & 1))
                atomicOr(p.status, CS_DEVICE_WAIT_TIMEOUT);
    } else if (warp == 1) {
        // ---------------------------------------------------------- MMA
        const uint64_t d0 = sw128_desc(smem_u32(smem));
        const uint32_t ta = tmem + kRACol;
        int s = 0;
        uint32_t use = 0, a_loads = 0;
        bool ok = true, new_m = true;
        auto advance = [&] {
            if (++s == kSlots) {
                s = 0;
                ++use;
            }
        };
        for (int tl = 0; tl < nt && ok; ++tl) {
            const int db = tl & 1;
            if (tl >= 2 && !wait_bar(&d_free[db], (uint32_t)((tl >> 1) - 1) & 1, p.status)) break;
            // the MMAs of the previous request tile are done with its rows
            if (new_m && a_loads > 0 && !wait_bar(a_free, (a_loads - 1) & 1, p.status)) break;
            const uint32_t td = tmem + db * kRN;
            const bool last_of_m = ++t == p.n_tiles;
            if (last_of_m) t = 0;
            if (new_m) {
                // the request tile's first group tile reads its rows from the
                // ring and leaves them in tensor memory for the next ones
                for (int kc = 0; kc < n_kc; ++kc) {
                    const int nb = p.n_boxes - kc * kStageBoxes;   // boxes left; a stage holds two at most
                    const int sa = s;
                    if (!(ok = wait_bar(&full[s], use & 1, p.status))) break;
                    advance();
                    if (!(ok = wait_bar(&full[s], use & 1, p.status))) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    if (elect_one()) {
                        const uint64_t da = d0 + (uint64_t)((sa * kStageBytes) >> 4);
                        const uint64_t ds = d0 + (uint64_t)((s * kStageBytes) >> 4);
                        const uint32_t tk = ta + kc * kStageBoxes * (kKC / 2);
                        const int steps = min(nb, kStageBoxes) * (kKC / 16);
#pragma unroll 1
                        for (int i = 0; i < steps; ++i) {
                            const uint64_t off = (uint64_t)(((i >> 2) * kBoxBytes) >> 4) + (i & 3) * 2;
                            tc_mma_ss(td, da + off, ds + off, route_idesc(), (kc > 0 || i > 0) ? 1u : 0u);
                        }
                        if (tl + 1 < nt) {
#pragma unroll 1
                            for (int i = 0; i < steps; ++i)
                                tc_cp_128x256b(tk + i * 8, da + (uint64_t)(((i >> 2) * kBoxBytes) >> 4) + (i & 3) * 2);
                        }
                        tc_commit(&empty[sa]);
                        tc_commit(&empty[s]);
                    }
                    __syncwarp();
                    advance();
                }
            } else {
                for (int kc = 0; kc < n_kc; ++kc) {
                    const int nb = p.n_boxes - kc * kStageBoxes;
                    if (!(ok = wait_bar(&full[s], use & 1, p.status))) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    if (elect_one()) {
                        // descriptors advance by whole boxes and 32-byte steps (addresses
                        // stay below 256 KB: the 14-bit start field cannot carry)
                        const uint64_t ds = d0 + (uint64_t)((s * kStageBytes) >> 4);
                        const uint32_t tk = ta + kc * kStageBoxes * (kKC / 2);
#pragma unroll
                        for (int k = 0; k < kStageBoxes; ++k) {
                            if (k >= nb) break;
#pragma unroll
                            for (int ks = 0; ks < kKC / 16; ++ks)
                                tc_mma_ts(td, tk + k * (kKC / 2) + ks * 8,
                                          ds + (uint64_t)((k * kBoxBytes) >> 4) + ks * 2, route_idesc(),
                                          (kc > 0 || k > 0 || ks > 0) ? 1u : 0u);
                        }
                        tc_commit(&empty[s]);
                    }
                    __syncwarp();
                    advance();
                }
            }
            if (!ok) break;
            if (elect_one()) {
                tc_commit(&d_full[db]);
                if (last_of_m) tc_commit(a_free);
            }
            __syncwarp();
            a_loads += new_m ? 1 : 0;
            new_m = last_of_m;
        }
        if (elect_one()) tc_commit(mma_done);
        __syncwarp();
        if (!mbar_wait_bounded(mma_done, 0)) atomicOr(p.status, CS_DEVICE_WAIT_TIMEOUT);
    } else if (warp >= 4) {
        // ------------------------------------------------------ epilogue
        const int sub = warp & 3, half = (warp - 4) >> 2;
        const int row = sub * 32 + lane;
        const uint32_t t_lane = tmem + ((uint32_t)(sub * 32) << 16) + half * (kRN / 2);
        const float kNaN = __int_as_float(0x7fffffff);   // excluded by fmaxf and by ==
        // this thread's share of the half's 64 inverse norms (warps 0 and 1 of it)
        const int col = half * (kRN / 2) + row;
        const bool loads = row < kRN / 2;
        auto inv_of = [&](int tile) {
            const int j = tile * kRN + col;
            return loads && j < p.N ? p.inv_norm_c[j] : kNaN;
        };
        float best = kNegInf;
        int idx = -1;
        auto flush = [&]() {
            if (half == 1) s_half[row] = make_float2(best, __int_as_float(idx));
            epi_sync();
            const int b = m * kRM + row;
            if (half == 0 && b < p.B) {
                const float2 o = s_half[row];
                const int oi = __float_as_int(o.y);
                if (oi >= 0 && (idx < 0 || o.x > best || (o.x == best && oi < idx))) {
                    best = o.x;
                    idx = oi;
                }
                const int slot = blockIdx.x - route_owner((long long)m * p.n_tiles, p.items, p.grid);
                p.part[((size_t)m * p.seg_slots + slot) * kRM + row] = make_float2(best, __int_as_float(idx));
            }
            epi_sync();
        };
        float inv_next = nt > 0 ? inv_of(t) : 0.f;
        bool dead = false;
        for (int tl = 0; tl < nt; ++tl) {
            const int db = tl & 1;
            float* inv = s_inv + db * kRN;
            if (loads) inv[col] = inv_next;
            epi_half_sync(half);
            const int tile = t;
            const bool last_of_m = ++t == p.n_tiles;
            if (last_of_m) t = 0;
            if (tl + 1 < nt) inv_next = inv_of(t);
            // after a timed-out wait the warp keeps taking part in the named
            // barriers but skips the rest
            // (a suspended wait: sixteen polling warps cost the issuing warps 10%)
            if (!dead && !__all_sync(0xffffffffu, mbar_wait_bounded(&d_full[db], (uint32_t)(tl >> 1) & 1))) {
                atomicOr(p.status, CS_DEVICE_WAIT_TIMEOUT);
                dead = true;
            }
            if (!dead) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                uint32_t r[2][32];
                tmem_ld32(r[0], t_lane + db * kRN);
                tmem_ld32(r[1], t_lane + db * kRN + 32);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&d_free[db]);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const float4* sv = reinterpret_cast<const float4*>(inv + half * (kRN / 2) + c * 32);
                    float sc[32];
                    float mx = kNegInf;
#pragma unroll
                    for (int q4 = 0; q4 < 8; ++q4) {
                        const float4 v = sv[q4];
                        sc[4 * q4 + 0] = __uint_as_float(r[c][4 * q4 + 0]) * v.x;
                        sc[4 * q4 + 1] = __uint_as_float(r[c][4 * q4 + 1]) * v.y;
                        sc[4 * q4 + 2] = __uint_as_float(r[c][4 * q4 + 2]) * v.z;
                        sc[4 * q4 + 3] = __uint_as_float(r[c][4 * q4 + 3]) * v.w;
                        mx = fmaxf(mx, fmaxf(fmaxf(sc[4 * q4], sc[4 * q4 + 1]), fmaxf(sc[4 * q4 + 2], sc[4 * q4 + 3])));
                    }
                    // ascending group ids and a strict > across chunks keep the
                    // lowest id of the maximum; inside the chunk, its first hit
                    if (mx > best) {
                        int e0 = 31;
#pragma unroll
                        for (int e = 31; e >= 0; --e)
                            if (sc[e] == mx) e0 = e;
                        best = mx;
                        idx = tile * kRN + half * (kRN / 2) + c * 32 + e0;
                    }
                }
            }
            if (last_of_m || tl == nt - 1) {
                flush();
                best = kNegInf;
                idx = -1;
                ++m;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 2)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kRTmemCols) : "memory");
}

// One warp per request: fold the partials of the CTAs that covered its
// request tile (higher score, then lower index), scale by the request's own
// inverse norm, apply the threshold.
__global__ void __launch_bounds__(256) route_merge_kernel(const __nv_bfloat16* emb, const float2* part, int B, int d,
                                                           int n_tiles, long long items, int grid, int seg_slots,
                                                           float tau, int32_t* out_group, int32_t* out_best,
                                                           float* out_score) {
    const int b = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    // the embeddings were complete before any CTA of the GEMM kernel let this
    // one start; without groups there is no such kernel in between
    if (n_tiles == 0) wait_prior_grid();
    float ss = 0.f;
    if (b < B) {
        __nv_bfloat16 e[kMaxRouteDim / 32];
#pragma unroll
        for (int j = 0; j < kMaxRouteDim / 32; ++j)
            e[j] = lane + 32 * j < d ? emb[(size_t)b * d + lane + 32 * j] : __float2bfloat16(0.f);
#pragma unroll
        for (int j = 0; j < kMaxRouteDim / 32; ++j) {
            const float x = __bfloat162float(e[j]);
            ss = fmaf(x, x, ss);
        }
    }
    wait_prior_grid();
    allow_dependent_launch();
    if (b >= B) return;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
    float best = kNegInf;
    int idx = -1;
    if (n_tiles > 0) {
        const int m = b / kRM;
        const int n_seg = route_owner((long long)(m + 1) * n_tiles - 1, items, grid) -
                          route_owner((long long)m * n_tiles, items, grid) + 1;
        for (int j = lane; j < n_seg; j += 32) {
            const float2 v = part[((size_t)m * seg_slots + j) * kRM + (b % kRM)];
            const int vi = __float_as_int(v.y);
            if (vi >= 0 && (idx < 0 || v.x > best || (v.x == best && vi < idx))) {
                best = v.x;
                idx = vi;
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, off);
        const int oi = __shfl_xor_sync(0xffffffffu, idx, off);
        if (oi >= 0 && (idx < 0 || ob > best || (ob == best && oi < idx))) {
            best = ob;
            idx = oi;
        }
    }
    if (lane == 0) {
        const float inv_e = ss > 0.f ? rsqrtf(ss) : 0.f;
        const float score = idx >= 0 ? best * inv_e : kNegInf;
        out_best[b] = idx;
        out_score[b] = score;
        out_group[b] = (idx >= 0 && score >= tau) ? idx : -1;
    }
}

// One warp per centroid: 1 / |c_i| (0 for a zero vector).
__global__ void __launch_bounds__(256) route_norms_kernel(const __nv_bfloat16* c, int N, int d, float* inv_norm) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= N) return;
    float ss = 0.f;
    for (int k = lane; k < d; k += 32) {
        const float x = __bfloat162float(c[(size_t)i * d + k]);
        ss = fmaf(x, x, ss);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
    if (lane == 0) inv_norm[i] = ss > 0.f ? rsqrtf(ss) : 0.f;
}

PFN_cuTensorMapEncodeTiled_v12000 route_encoder() {
    static std::atomic<PFN_cuTensorMapEncodeTiled_v12000> fn{nullptr};
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
    }
    return fn;
}

// [rows, d] bf16 row-major as (d, rows); box {64, 128}, 128-byte swizzle.
cs_status encode_rows_map(CUtensorMap* map, const void* base, int rows, int d) {
    auto enc = route_encoder();
    if (!enc) return fail(CS_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    const cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)(rows > 0 ? rows : 1)};
    const cuuint64_t strides[1] = {(cuuint64_t)d * 2};
    const cuuint32_t box[2] = {kKC, kRM};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
                           estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(CS_ERR_CUDA, "cuTensorMapEncodeTiled(route) failed (CUresult %d)", (int)r);
    return CS_OK;
}

}  // namespace

RoutePlan plan_route(const cs_route_dims& d, int sm_count) {
    RoutePlan pl{};
    pl.m_tiles = (d.batch + kRM - 1) / kRM;
    pl.n_tiles = (d.n_groups + kRN - 1) / kRN;
    pl.items = (long long)pl.m_tiles * pl.n_tiles;
    const int sms = sm_count > 0 ? sm_count : 148;
    pl.grid = (int)(pl.items < sms ? pl.items : sms);
    // CTAs covering one request tile: its n_tiles items meet at most
    // floor((n_tiles - 1) * G / I) + 2 of the G ranges
    pl.seg_slots = pl.items > 0 ? (int)(((long long)(pl.n_tiles - 1) * pl.grid) / pl.items) + 2 : 0;
    pl.bytes = 256 + ((size_t)pl.m_tiles * pl.seg_slots * kRM * sizeof(float2) + 255) / 256 * 256;
    return pl;
}

cs_status launch_route(const cs_route_dims& d, const RoutePlan& pl, const void* emb, const void* centroids,
                       const float* inv_norms, float tau, int32_t* out_group, int32_t* out_best,
                       float* out_score, void* workspace, cudaStream_t stream) {
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    cudaError_t e;
    if (pl.grid > 0) {
        CUtensorMap te, tc;
        cs_status st = encode_rows_map(&te, emb, d.batch, d.dim);
        if (st != CS_OK) return st;
        st = encode_rows_map(&tc, centroids, d.n_groups, d.dim);
        if (st != CS_OK) return st;
        static std::atomic<bool> attr_set[64];
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev < 0 || dev >= 64 || !attr_set[dev]) {
            e = cudaFuncSetAttribute(route_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kRSmemBytes);
            if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(route_gemm_kernel)");
            if (dev >= 0 && dev < 64) attr_set[dev] = true;
        }
        RouteParams p{};
        p.B = d.batch;
        p.N = d.n_groups;
        p.n_boxes = d.dim / kKC;
        p.n_tiles = pl.n_tiles;
        p.grid = pl.grid;
        p.seg_slots = pl.seg_slots;
        p.items = pl.items;
        p.inv_norm_c = inv_norms;
        p.status = reinterpret_cast<int*>(ws);
        p.part = reinterpret_cast<float2*>(ws + 256);
        e = launch_dependent(route_gemm_kernel, dim3(pl.grid), dim3(kRThreads), kRSmemBytes, stream, te, tc, p);
        if (e != cudaSuccess) return cuda_fail(e, "route_gemm_kernel launch");
    }
    e = launch_dependent(route_merge_kernel, dim3((d.batch + 7) / 8), dim3(256), 0, stream,
                         static_cast<const __nv_bfloat16*>(emb), reinterpret_cast<const float2*>(ws + 256), d.batch,
                         d.dim, pl.n_tiles, pl.items, pl.grid, pl.seg_slots, tau, out_group, out_best, out_score);
    if (e != cudaSuccess) return cuda_fail(e, "route_merge_kernel launch");
    return CS_OK;
}

cs_status launch_route_norms(int n_groups, int dim, const void* centroids, float* inv_norms, cudaStream_t stream) {
    route_norms_kernel<<<(n_groups + 7) / 8, 256, 0, stream>>>(static_cast<const __nv_bfloat16*>(centroids),
                                                               n_groups, dim, inv_norms);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "route_norms_kernel launch");
    return CS_OK;
}

}  // namespace cs
