// spec_accept_walk.cuh -- the walk and the draw of the acceptance step
// (included by spec_accept.cu inside its anonymous namespace, whose row
// helpers it shares).
//
// One thread-block cluster per request walks its draft: a chain is the tree
// in which node u's only child is u + 1, the sampler a tree of one node, so
// all of them run this kernel.
//  * After accept_stats_kernel (kStream = false) the statistics of the rows
//    are folded from its partials, or a phase's test has decided already.
//  * kStream = true, trees: no kernel has run before.  In a round the cluster
//    streams the target and draft rows of the next undecided node, swaps the
//    row statistics through distributed shared memory and walks on; the walk
//    usually stops early, and the rows past it are never read.
// The draw: where the unit masses of the row (pair) are known they are the
// CDF, and one CTA weighs the unit that holds the cell.  Otherwise the cluster
// weighs the whole pair, 1 KB blocks of it dealt over its warps, and swaps the
// slice masses.  One warp then walks the block that holds the cell.
// What bounds a call of this size is latency, and of that a good part is
// instruction fetches (ncu: 8 to 14 cycles an issue waiting for instructions
// in a form with every loop unrolled, B = 8): hence the rolled loops, the one
// weighing routine for p and max(p - kappa q, 0), and the row ends in one
// out-of-line routine.  B = 8, k = 5, V = 128256: 19.6 -> 14.9 us a call.
//
// Blocks start at 16-byte boundaries of memory, so rows of any alignment take
// vector loads; CTA `rank` of a cluster owns blocks [rank * per, (rank + 1) *
// per) of every row.

constexpr int kWalkMaxThreads = 256;
constexpr int kWalkMaxWarps = kWalkMaxThreads / 32;
constexpr int kWalkVecs = 4;                   // streaming: 16-byte vectors per lane per block (2 KB of a row)
constexpr int kRunVecs = 2;                    // draw: contiguous vectors per lane per block (1 KB of a row)
constexpr int kWalkSegs = 2050;                // draw blocks of one row per CTA, at most

struct WalkParams {
    const void* target;       // [B, n, V]
    const void* draft;        // [B, d_rows, V]: chain d_rows = n - 1, tree n (null when greedy or n = 1)
    const int32_t* tokens;    // chain [B, n-1]: node c's token is tokens[c-1]; tree [B, n]
    const float* uniforms;    // [B, n]: u_{c-1} tests node c, u_{n-1} is the draw
    const int32_t* parents;   // tree [B, n]; null for the chain
    int32_t* out_tokens;      // [B, n]
    int32_t* out_n;           // [B], or null (the sampler)
    int32_t* out_path;        // tree [B, n]
    int B, V, n, d_rows;
    int I;                    // 4 KB items of a row (accept_stats_kernel's)
    int blocks, per;          // 2 KB blocks of a row, blocks of a row per CTA
    Phase ph;                 // the last phase of accept_stats_kernel (R == 0: it did not run)
    Decided dec;              // what the earlier phases decided (read when ph.undecided is set),
    const float* mass;        // and [B, units] the draw masses of the units of the pair that decided
    int b_base;               // first request of this launch
    float c_hi, c_lo;         // log2(e) / T as a float pair
};

template <typename T>
struct RunPair {   // one lane's run of a draw block: kRunVecs contiguous vectors of both rows
    uint4 t[kRunVecs], d[kRunVecs];
};

// Draw block j (32 runs) of the row pair, in the target row's blocks.
template <typename T>
__device__ __forceinline__ void load_run(const DrawRow<T>& d, int j, int V, int lane, RunPair<T>& r) {
    constexpr int kPer = 16 / (int)sizeof(T), kBlock = 32 * kRunVecs * kPer;
    const int base = j * kBlock - misaligned_by(d.rt);
    load_pair(d.rt, d.rd, d.same, base, kBlock, base + lane * kRunVecs * kPer, kPer, V, r.t, r.d);
}

template <typename T>
__device__ __forceinline__ void weigh_run(const DrawRow<T>& d, const RunPair<T>& r,
                                          float (&w)[kRunVecs * 16 / sizeof(T)]) {
#pragma unroll
    for (int u = 0; u < kRunVecs; ++u) weigh(d, r.t[u], r.d[u], w + u * (16 / (int)sizeof(T)));
}

// Mass of each of the draw blocks [j0, j0 + nj) of row pair d into s_seg
// (warp w takes every nw-th); two blocks are in flight while one is summed.
template <typename T>
__device__ __forceinline__ void walk_masses(const DrawRow<T>& d, int j0, int nj, int V, float* s_seg) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    int j = threadIdx.x >> 5;
    RunPair<T> cur, nx1, nx2;
    if (j < nj) load_run(d, j0 + j, V, lane, cur);
    if (j + nw < nj) load_run(d, j0 + j + nw, V, lane, nx1);
#pragma unroll 1
    for (; j < nj; j += nw) {
        if (j + 2 * nw < nj) load_run(d, j0 + j + 2 * nw, V, lane, nx2);
        float w[kRunVecs * 16 / sizeof(T)];
        weigh_run(d, cur, w);
        float acc = 0.f;
#pragma unroll
        for (int e = 0; e < kRunVecs * 16 / (int)sizeof(T); ++e) acc += w[e];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (lane == 0) s_seg[j] = acc;
        cur = nx1;
        nx1 = nx2;
    }
}

// The token of draw block j where the running mass passes `rem` (through
// rounding: the block's last one of positive weight), by one warp; -1 when
// no weight is positive.
template <typename T>
__device__ __forceinline__ int walk_locate(const DrawRow<T>& d, int j, int V, float rem) {
    constexpr int kPer = 16 / (int)sizeof(T), kRun = kRunVecs * kPer;
    const int lane = threadIdx.x & 31;
    const int at = (j * 32 + lane) * kRun - misaligned_by(d.rt);
    RunPair<T> r;
    load_run(d, j, V, lane, r);
    float w[kRun];
    weigh_run(d, r, w);
    float own = 0.f;
    int last = -1;
#pragma unroll
    for (int e = 0; e < kRun; ++e) {
        own += w[e];
        if (w[e] > 0.f) last = at + e;
    }
    const float incl = warp_incl_scan(own, lane);
    float c = incl - own;
    int pick = -1;
#pragma unroll
    for (int e = 0; e < kRun; ++e) {
        c += w[e];
        if (w[e] > 0.f && pick < 0 && c > rem) pick = at + e;
    }
    // only a run with positive mass can own the draw; a run that passes rem by
    // its scan but by no running sum of its own owns it with its last weight
    const unsigned hit = __ballot_sync(0xffffffffu, own > 0.f && incl > rem);
    if (hit) return __shfl_sync(0xffffffffu, pick >= 0 ? pick : last, __ffs(hit) - 1);
    return warp_max_int(last);
}

// A sum and its rounding error (h the nearest float to h + l): the two-sum of
// Knuth, kept as a double-length number as Dekker (1971) does.
struct Sum2 {
    float h, l;
};

__device__ __forceinline__ Sum2 add2(Sum2 a, Sum2 b) {
    const float s = a.h + b.h, bb = s - a.h;
    const float e = ((a.h - (s - bb)) + (b.h - bb)) + (a.l + b.l);
    const float h = s + e;
    return {h, e - (h - s)};
}

__device__ __forceinline__ Sum2 shfl2(Sum2 v, int src) {
    return {__shfl_sync(0xffffffffu, v.h, src), __shfl_sync(0xffffffffu, v.l, src)};
}

__device__ __forceinline__ Sum2 sub2(Sum2 a, Sum2 b) { return add2(a, {-b.h, -b.l}); }

// u times a sum.
__device__ __forceinline__ Sum2 scale2(float u, Sum2 z) {
    const float p = u * z.h;
    return add2({p, 0.f}, {fmaf(u, z.h, -p), u * z.l});
}

// Inclusive scan of the warp's values (out of line: one copy of its steps to
// fetch; lanes below a step's distance add zero).
__device__ __noinline__ Sum2 warp_incl_scan2(Sum2 v, int lane) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const float h = __shfl_up_sync(0xffffffffu, v.h, off), l = __shfl_up_sync(0xffffffffu, v.l, off);
        v = add2(v, {lane >= off ? h : 0.f, lane >= off ? l : 0.f});
    }
    return v;
}

// Writes v to the same shared-memory address of CTA `rank` of the cluster.
__device__ __forceinline__ void st_cluster_f2(float2* local, uint32_t rank, float2 v) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(local)), "r"(rank));
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(remote), "f"(v.x), "f"(v.y) : "memory");
}

// Every CTA of the cluster past this point sees what the others wrote before it.
__device__ __forceinline__ void walk_sync(uint32_t n_ranks) {
    if (n_ranks > 1) {
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }
}

template <typename T, bool kGreedy, bool kStream>
__global__ void __launch_bounds__(kWalkMaxThreads, 2) accept_walk_kernel(const WalkParams p) {
    constexpr int kPer = 16 / (int)sizeof(T);
    constexpr int kBlock = 32 * kWalkVecs * kPer;
    __shared__ unsigned long long s_kids[kMaxTreeNodes];
    __shared__ float2 s_stat[2 * kMaxTreeNodes];             // row statistics: 2 node (target), 2 node + 1 (draft)
    __shared__ float2 s_z[kMaxTreeNodes];                    // target / draft logit of node c's token in its parent's rows
    __shared__ int s_tok[kMaxTreeNodes], s_path[kMaxTreeNodes];
    __shared__ float s_u[kMaxTreeNodes];
    __shared__ float2 s_part[2][kWalkMaxWarps];              // a round's statistics per row (target, draft) and warp
    __shared__ float2 s_x[2][2][kMaxCluster];                // ... per row and CTA, by round parity
    __shared__ float s_seg[kWalkSegs], s_cum[kWalkSegs];     // draw masses of the blocks and their running sum
    __shared__ float2 s_m[2][kMaxCluster];                   // draw mass per CTA

    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5, nth = blockDim.x;
    const uint32_t rank = cluster_rank(), n_ranks = cluster_size();
    // (the requests whose rows were read last come first: they are the
    // likeliest to be in L2 still)
    const int b = p.b_base + (int)(gridDim.y - 1 - blockIdx.y);
    const int n = p.n, V = p.V;
    const bool tree = p.parents != nullptr;
    const float2 empty = make_float2(kNegInf, kGreedy ? __int_as_float(INT_MAX) : 0.f);
    if (n_ranks > 1) cluster_arrive();   // met by the wait before the first remote write
    bool started = n_ranks == 1;
    if (kStream) {
        // the first kernel of its call: nothing is read before the kernel before it is done
        wait_prior_grid();
        allow_dependent_launch();   // the next kernel may start (it waits for this grid before it reads its results)
    }

    const T* const target = static_cast<const T*>(p.target) + (size_t)b * n * V;
    const T* const draft = static_cast<const T*>(p.draft) + (size_t)b * p.d_rows * V;

    // ---- the draft: thread c < n (n <= 64 <= threads) holds node c
    int par = -1, tok = -1;
    if (tid < n) {
        if (tree) {
            const int q = tid > 0 ? p.parents[(size_t)b * n + tid] : -1;
            par = q >= 0 && q < tid ? q : -1;
            tok = p.tokens[(size_t)b * n + tid];
        } else if (tid > 0) {
            par = tid - 1;
            tok = p.tokens[(size_t)b * (n - 1) + tid - 1];
        }
        if (!kGreedy) s_u[tid] = p.uniforms[(size_t)b * n + tid];
        s_tok[tid] = tok;
        s_kids[tid] = tree || tid + 1 == n ? 0ull : 1ull << (tid + 1);
    }
    if (tree) {
        __syncthreads();
        if (tid < n && par >= 0) atomicOr(&s_kids[par], 1ull << tid);
    }
    // the logits that its tests need (an invalid token tests as ratio 0); called once
    float2 z = make_float2(kNegInf, 0.f);
    auto load_tests = [&]() {
        if (!kGreedy && tid < n && par >= 0 && tok >= 0 && tok < V) {
            z.x = to_f(target[(size_t)par * V + tok]);
            z.y = to_f(draft[(size_t)par * V + tok]);
        }
    };
    bool first = true;

    const int j0 = (int)rank * p.per;                        // this CTA's blocks of every row
    const int nj = max(0, min(p.per, p.blocks - j0));
    constexpr int kSub = kWalkVecs / kRunVecs;               // draw blocks per streaming block
    uint64_t have = 0;
    int node = 0, depth = 0, xr = 0, xm = 0, emit = 0;
    float kappa = 0.f;
    bool decided = false;
    if (!kStream) {
        load_tests();
        if (tid < n) {
            s_z[tid] = z;
            s_path[tid] = tid + 1;   // a chain's (a tree's is written as it is walked)
        }
        first = false;
        wait_prior_grid();
        allow_dependent_launch();
        node = depth = p.ph.p0;
        have = (p.ph.t_rows < 64 ? (1ull << p.ph.t_rows) - 1ull : ~0ull) << p.ph.p0;
        if (p.ph.undecided) {
            // (every request is decided: the calls read in phases end with one more
            // test; the bounds are for a workspace that another call writes at the
            // same time, whose tokens are undefined but whose reads are not)
            const int a = max(0, min(__ldcg(p.dec.a + b), n - 1));
            const float4 st = __ldcg(p.dec.stat + b);
            decided = true;
            node = depth = a;
            kappa = a + 1 < n ? 1.f : 0.f;
            emit = __float_as_int(st.x);
            if (tid == 0) {
                s_stat[2 * a] = make_float2(st.x, st.y);
                s_stat[2 * a + 1] = make_float2(st.z, st.w);
            }
        }
        if (!decided) {
            // bit-identical in every CTA of the cluster
            constexpr int kBatch = 2;
            const int R = p.ph.R, g = p.ph.t_rows;
#pragma unroll 1
            for (int r0 = wid; r0 < R; r0 += kBatch * nw) {
                float2 f[kBatch];
                fold_rows<kGreedy, kBatch>(p.ph, b, r0, nw, lane, p.c_hi, p.c_lo, f);
#pragma unroll
                for (int i = 0; i < kBatch; ++i) {
                    const int r = r0 + i * nw;
                    if (lane == i && r < R) s_stat[2 * p.ph.p0 + (r < g ? 2 * r : 2 * (r - g) + 1)] = f[i];
                }
            }
        }
        __syncthreads();
    }

    DrawRow<T> d;
    // the weights of node u's rows at kappa
    auto set_pair = [&](int u, float kap) {
        d.rt = target + (size_t)u * V;
        d.rd = draft + (size_t)u * V;
        set_weights(d, s_stat[2 * u], s_stat[2 * u + 1], kap, p.c_hi);
    };
    // the running sum of `count` item masses into s_cum (by warp 0); their total
    auto sum_items = [&](int count) -> float {
        float tot = 0.f;
#pragma unroll 1
        for (int q0 = 0; q0 < count; q0 += 32) {
            const float inc = warp_incl_scan(q0 + lane < count ? s_seg[q0 + lane] : 0.f, lane);
            if (wid == 0 && q0 + lane < count) s_cum[q0 + lane] = tot + inc;
            tot += __shfl_sync(0xffffffffu, inc, 31);
        }
        return tot;
    };
    // masses of this CTA's items summed and swapped: the mass of rank `lane`
    // (zero past the last rank)
    auto swap_mass = [&]() -> float {
        const float tot = sum_items(nj * kSub);
        if (n_ranks == 1) return lane == 0 ? tot : 0.f;
        if (!started) {   // every CTA of the cluster runs: its shared memory may be written
            cluster_wait();
            started = true;
        }
        const int slot = xm++ & 1;
        if (wid == 0 && lane < (int)n_ranks) st_cluster_f2(&s_m[slot][rank], lane, make_float2(tot, 0.f));
        walk_sync(n_ranks);
        return lane < (int)n_ranks ? s_m[slot][lane].x : 0.f;
    };

    bool stop = decided;
    if (!kStream && !tree && !stop) {
        // a chain's last phase: lane i of every warp tests position node + i
        const int at = node + lane;
        bool rej = false;
        int top = 0;
        if (at < n) {
            const float2 st = s_stat[2 * at];
            if (kGreedy) {
                top = __float_as_int(st.y);
                if (top == INT_MAX) top = 0;   // a row with no finite entry
            }
            if (at + 1 < n) {
                if (kGreedy) {
                    rej = s_tok[at + 1] != top;
                } else {
                    const float2 zc = s_z[at + 1];
                    rej = !(s_u[at] < accept_ratio(zc.x != kNegInf, zc.x, zc.y, st, s_stat[2 * at + 1], p.c_hi, p.c_lo));
                }
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, rej);
        if (m) kappa = 1.f;
        node = depth = m ? node + __ffs(m) - 1 : n - 1;
        emit = __shfl_sync(0xffffffffu, top, node - p.ph.p0);
        stop = true;
    }
    while (!stop) {
        if (kStream && !((have >> node) & 1ull)) {
            // ---- a round: the rows of the current node (a leaf's draft row is not read)
            __syncthreads();   // s_kids complete; the last round's s_part are no longer read
            const int n_rows = kGreedy || !s_kids[node] ? 1 : 2;
            have |= 1ull << node;

            // ---- row statistics: the flattened items of the rows, dealt over the warps
            if (lane < n_rows) s_part[lane][wid] = empty;
            __syncwarp();
            auto row_of = [&](int r) -> const T* { return (r ? draft : target) + (size_t)node * V; };
            const int total = n_rows * nj;
            int idx = wid, r = nj > 0 ? wid / nj : 0, j = nj > 0 ? wid - r * nj : 0;
            uint4 cur[kWalkVecs], nxt[kWalkVecs];
            if (idx < total) load_block(row_of(r), j0 + j, V, lane, cur);
            if (first) load_tests();
            float m = kNegInf, s = 0.f;
            int id = INT_MAX;
#pragma unroll 1
            while (idx < total) {
                const int nidx = idx + nw;
                int nr = r, njj = j + nw;
                while (njj >= nj) {
                    njj -= nj;
                    ++nr;
                }
                if (nidx < total) load_block(row_of(nr), j0 + njj, V, lane, nxt);
                if (kGreedy) {
                    item_argmax<T>(cur, (j0 + j) * kBlock - misaligned_by(row_of(r)) + lane * kPer, m, id);
                } else {
                    const float mi = item_max(cur, T());
                    if (mi > m) {
                        s = m == kNegInf ? 0.f : s * ex2_scaled(m - mi, p.c_hi, p.c_lo);
                        m = mi;
                    }
                    if (m != kNegInf) s += item_sum<T>(cur, m, p.c_hi);
                }
                if (nr != r || nidx >= total) {
                    const float2 f = kGreedy ? warp_fold_argmax(make_float2(m, __int_as_float(id)))
                                             : warp_fold_sum(m, s, p.c_hi, p.c_lo);
                    if (lane == 0) s_part[r][wid] = f;
                    m = kNegInf;
                    s = 0.f;
                    id = INT_MAX;
                }
                idx = nidx;
                r = nr;
                j = njj;
#pragma unroll
                for (int u = 0; u < kWalkVecs; ++u) cur[u] = nxt[u];
            }
            if (first && tid < n) s_z[tid] = z;
            first = false;
            if (!started) {
                cluster_wait();
                started = true;
            }
            __syncthreads();
            const int slot = xr++ & 1;
#pragma unroll 1
            for (int q = wid; q < n_rows; q += nw) {
                float2 f = lane < nw ? s_part[q][lane] : empty;
                f = kGreedy ? warp_fold_argmax(f) : warp_fold_sum(f.x, f.y, p.c_hi, p.c_lo);
                if (n_ranks == 1) {
                    if (lane == 0) s_stat[2 * node + q] = f;
                } else if (lane < (int)n_ranks) {
                    st_cluster_f2(&s_x[slot][q][rank], lane, f);
                }
            }
            if (n_ranks > 1) {
                walk_sync(n_ranks);
                // every CTA folds the ranks in the same order: bit-identical statistics
#pragma unroll 1
                for (int q = wid; q < n_rows; q += nw) {
                    float2 f = lane < (int)n_ranks ? s_x[slot][q][lane] : empty;
                    f = kGreedy ? warp_fold_argmax(f) : warp_fold_sum(f.x, f.y, p.c_hi, p.c_lo);
                    if (lane == 0) s_stat[2 * node + q] = f;
                }
            }
            __syncthreads();
        }

        // ---- the walk, as far as the statistics reach: every thread of the
        // cluster takes the same decisions from the same numbers
#pragma unroll 1
        while ((have >> node) & 1ull) {
            int next = -1;
            unsigned long long kids = s_kids[node];
            if (kGreedy) {
                emit = __float_as_int(s_stat[2 * node].y);
                if (emit == INT_MAX) emit = 0;   // a row with no finite entry
                while (kids && next < 0) {
                    const int c = __ffsll((long long)kids) - 1;
                    kids &= kids - 1;
                    if (s_tok[c] == emit) next = c;
                }
            } else {
                // node c with token x is accepted iff u_{c-1} < max(p(x)/q(x) -
                // kappa, 0) / Z; a rejection adds Z to kappa, and the residual
                // max(p - kappa q, 0) has to be summed only if a sibling follows
                const float2 st = s_stat[2 * node], sd = s_stat[2 * node + 1];
                float kap = 0.f, Z = 1.f;
#pragma unroll 1
                while (kids) {
                    const int c = __ffsll((long long)kids) - 1;
                    kids &= kids - 1;
                    const float2 zc = s_z[c];
                    float ratio = accept_ratio(zc.x != kNegInf, zc.x, zc.y, st, sd, p.c_hi, p.c_lo);
                    if (kap > 0.f) ratio = fmaxf(ratio - kap, 0.f) / Z;
                    if (s_u[c - 1] < ratio) {
                        next = c;
                        break;
                    }
                    kap += Z;
                    if (!kids) break;
                    set_pair(node, kap);
                    walk_masses(d, j0 * kSub, nj * kSub, V, s_seg);
                    __syncthreads();
                    Z = __shfl_sync(0xffffffffu, warp_incl_scan(swap_mass(), lane), 31) / st.y;
                    __syncthreads();   // s_seg is no longer read
                    if (!(Z > 0.f)) {   // no positive residual (p == kappa q up to rounding): draw from p
                        kap = 0.f;
                        break;
                    }
                }
                if (next < 0) kappa = kap;
            }
            if (next < 0) {
                stop = true;
                break;
            }
            if (tid == 0) s_path[depth] = next;
            ++depth;
            node = next;
        }
    }
    __syncthreads();   // s_path

    // ---- the draw from max(p - kappa q, 0), or from p
    int token = emit, writer = kGreedy && rank == 0 ? 0 : -1;
    if (!kGreedy) {
        const float kInf = __int_as_float(0x7f800000);
        const float uk = s_u[n - 1];
        bool residual = kappa > 0.f;
        set_pair(node, kappa);
        // the draw blocks [jb, jb + count) whose masses are in s_seg, the mass
        // tt past their start, and whether this CTA finds the token there
        int jb = j0 * kSub, count = nj * kSub;
        float tt = kInf;
        bool mine = false;
        int i0 = 0, i1 = 0;
        if (!kStream && (!residual || decided)) {
            // the unit masses are known -- of a row of the statistics kernel,
            // drawn from without a residual, or of a pair decided in an earlier
            // phase: they are the CDF, and one CTA weighs the unit that holds
            // the cell
            const float2* part = p.ph.part + ((size_t)b * p.ph.R + (node - p.ph.p0)) * p.ph.units;
            auto mass = [&](int l) {
                if (l >= p.ph.units) return 0.f;
                if (residual) return __ldcg(p.mass + (size_t)b * p.ph.units + l);
                const float2 f = __ldcg(part + l);
                const float x = f.x == kNegInf ? 0.f : f.y * ex2_scaled(f.x - d.mt, p.c_hi, p.c_lo);
                return x > 0x1p-120f ? x : 0.f;   // a unit that counts has a weight that is not flushed
            };
            // the CDF over the units and the draw's place in it as pairs of
            // floats: a token of 1e-6 of the mass is 16 roundings of a float
            // sum (against 64 bits 14 of 5872 draws moved to the next token,
            // 4 with pairs; in doubles 256 rows of 128256 took 1.5 us longer)
            const float x0 = mass(lane);
            const Sum2 incl0 = warp_incl_scan2({x0, 0.f}, lane);
            Sum2 Z = shfl2(incl0, 31);
#pragma unroll 1
            for (int l0 = 32; l0 < p.ph.units; l0 += 32) Z = add2(Z, shfl2(warp_incl_scan2({mass(l0 + lane), 0.f}, lane), 31));
            // u Z, less the units passed
            Sum2 rest = scale2(uk, Z);
            int at = -1, last = -1;
#pragma unroll 1
            for (int l0 = 0; l0 < p.ph.units && at < 0; l0 += 32) {
                const float x = l0 > 0 ? mass(l0 + lane) : x0;
                const Sum2 incl = l0 > 0 ? warp_incl_scan2({x, 0.f}, lane) : incl0;
                const Sum2 past = sub2(incl, rest);
                const unsigned hit = __ballot_sync(0xffffffffu, x > 0.f && past.h > 0.f);
                const unsigned any = __ballot_sync(0xffffffffu, x > 0.f);
                if (hit) {
                    at = l0 + __ffs(hit) - 1;
                    tt = __shfl_sync(0xffffffffu, sub2({x, 0.f}, past).h, at - l0);
                }
                if (any) last = l0 + 31 - __clz((int)any);
                rest = sub2(rest, shfl2(incl, 31));
            }
            if (at < 0) at = last;   // past the total through rounding: the last positive unit (tt: its end)
            if (at >= 0) {           // (no mass at all: the residual is empty up to rounding, drawn from p below)
                i0 = at * p.ph.U;
                i1 = min(i0 + p.ph.U, p.I);
            } else {
                residual = false;
                set_pair(node, 0.f);
            }
        }
        constexpr int kItemSubs = kVecs / kRunVecs;   // draw blocks per item
        const bool one = i1 > i0 && (i1 - i0) * kItemSubs <= kWalkSegs;
        if (one) {
            jb = i0 * kItemSubs;
            count = rank == 0 ? (i1 - i0) * kItemSubs : 0;
            mine = rank == 0;
        }
        if (count > 8 * nw) {
            // many blocks a warp: ask L2 for the slice now (only addresses inside the rows)
            constexpr int kLine = 128 / (int)sizeof(T);
            const int e0 = jb * (32 * kRunVecs * kPer), e1 = min(V, e0 + count * (32 * kRunVecs * kPer));
            for (int e = e0 + tid * kLine; e < e1; e += nth * kLine) {
                asm volatile("prefetch.global.L2 [%0];" ::"l"(d.rt + e));
                if (residual) asm volatile("prefetch.global.L2 [%0];" ::"l"(d.rd + e));
            }
        }
#pragma unroll 1
        for (;;) {
            walk_masses(d, jb, count, V, s_seg);
            __syncthreads();
            if (one) {
                sum_items(count);
                break;
            }
            const float x = swap_mass();
            const Sum2 incl = warp_incl_scan2({x, 0.f}, lane), Z = shfl2(incl, 31);
            if (Z.h > 0.f || !residual) {
                // the CTA whose cell holds u Z (past the total through rounding: the last positive mass)
                const Sum2 past = sub2(incl, scale2(uk, Z));
                const unsigned own = __ballot_sync(0xffffffffu, x > 0.f && past.h > 0.f);
                const unsigned pos = __ballot_sync(0xffffffffu, x > 0.f);
                const int owner = own ? __ffs(own) - 1 : pos ? 31 - __clz((int)pos) : 0;
                mine = (int)rank == owner;
                if (own) tt = __shfl_sync(0xffffffffu, sub2({x, 0.f}, past).h, owner);
                break;
            }
            residual = false;   // no positive residual (p == q up to rounding): draw from p instead
            set_pair(node, 0.f);
            __syncthreads();    // s_seg is no longer read
        }
        if (mine && wid == 0) {
            __syncwarp();
            int seg = -1, last = -1;
#pragma unroll 1
            for (int q0 = 0; q0 < count && seg < 0; q0 += 32) {
                const bool in = q0 + lane < count && s_seg[q0 + lane] > 0.f;
                const unsigned hit = __ballot_sync(0xffffffffu, in && s_cum[q0 + lane] > tt);
                const unsigned any = __ballot_sync(0xffffffffu, in);
                if (hit) seg = q0 + __ffs(hit) - 1;
                if (any) last = q0 + 31 - __clz((int)any);
            }
            const float rem = seg > 0 ? tt - s_cum[seg - 1] : seg == 0 ? tt : kInf;
            if (seg < 0) seg = last;   // through rounding: the last block of positive mass
            token = seg >= 0 ? max(walk_locate(d, jb + seg, V, rem), 0) : 0;
            writer = 0;
        }
    }
    int32_t* out = p.out_tokens + (size_t)b * n;
    if (tid == writer) out[depth] = token;
    if (rank == 0) {
        for (int i = tid; i < n; i += nth) {
            if (i < depth) out[i] = s_tok[s_path[i]];
            else if (i > depth) out[i] = -1;
            if (tree) p.out_path[(size_t)b * n + i] = i < depth ? s_path[i] : -1;
        }
        if (tid == 0 && p.out_n) p.out_n[b] = depth;
    }
    // a remote write meets a CTA that still runs: every one is followed by a
    // cluster barrier; the barrier of the start is met here if no row was swapped
    if (!started) {
        __syncthreads();
        cluster_wait();
    }
}
