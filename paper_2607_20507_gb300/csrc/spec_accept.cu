// spec_accept.cu -- the acceptance step of speculative sampling (the rule
// the paper's drafter follows, Sec. 3.4): temperature softmax statistics of
// target and draft rows, the min(1, p/q) accept test, the residual
// max(0, p - q) or bonus draw by inverse CDF, and the greedy variant.
//
// Kernels of a call, each a programmatic dependent of the one before it (no
// spin-waits, no scratch that has to start at a known value):
//   1. accept_stats_kernel streams rows of every request (target rows, then
//      draft rows; target rows only when greedy) once.  Rows are cut into 4 KB
//      items and units of a few items; a warp keeps the next item in flight
//      while it reduces the current one and writes one partial per unit: (max,
//      sum 2^((z-max)c)) -- one exponential per logit -- or, greedy, (max,
//      lowest id of the max).
//   2. accept_walk_kernel, one thread-block cluster per request, folds the
//      partials of the request's rows (every CTA in the same order, so all of
//      them hold bit-identical statistics), runs the accept tests (one lane
//      per position, the first rejection found by a ballot) and draws: the
//      masses of the CTAs' slices of the deciding row pair are swapped through
//      distributed shared memory, and one warp of the CTA whose cell holds
//      u_k * Z finds the token.  Greedy: the arg max of the deciding row.
// A chain's rows past its first rejection are not needed, so a call that
// takes long to read (plan_accept) reads its positions in phases: kernel 1 for
// the first positions of every request, accept_test_kernel for their tests,
// kernel 1 for the next positions of the requests that are still undecided
// (and for the draw masses of those just decided, whose rows are still in
// L2), and so on; the walk then only draws.
// Token trees (multi-candidate verification) walk likewise: the children of
// the current node are tested in turn, each rejection turning the running
// distribution into the residual max(p - kappa q, 0) / Z, whose mass Z takes
// one cluster-wide pass over the row pair.  A large tree skips kernel 1: the
// walk streams the rows of the nodes that it comes to.
// No probability is written to memory; the scratch holds the units' partials,
// draw masses and the phases' decisions.
#include <limits.h>
#include <math.h>

#include "cs_device.cuh"
#include "cs_internal.h"

namespace cs {
namespace {

constexpr int kThreads = 256;                  // the statistics kernel
constexpr int kWarps = kThreads / 32;
constexpr int kVecs = 8;                       // 16-byte vectors per lane per item
constexpr int kItemBytes = 32 * kVecs * 16;    // 4 KB of one row
constexpr int kMaxCluster = 16;
constexpr int kMaxTreeNodes = 64;
constexpr int kMaxPhased = 4096;               // requests of a call whose positions are read in phases, at most

// x / d for 0 <= x by a multiplication whenever x < 2^31 (division by an
// invariant integer, Granlund and Montgomery 1994): with
// s = ceil(log2 d) and mul = floor(2^(31+s) / d) + 1 < 2^32 + 1, the error of
// x mul / 2^(31+s) over x / d is below x / 2^(31+s) < 1/d, too little to reach
// the next whole number.
struct FastDiv {
    long long d;
    unsigned long long mul;
    int shift;
    __host__ void set(long long by) {
        if (by < 1) by = 1;
        d = by;
        shift = 31;
        while ((1ll << (shift - 31)) < by) ++shift;
        mul = (1ull << shift) / (unsigned long long)by + 1;
    }
    __device__ __forceinline__ long long div(long long x) const {
        return x < 0x80000000ll ? (long long)((unsigned long long)x * mul >> shift) : x / d;
    }
};

// The rows that one launch of the statistics kernel reads, and where their
// partials are.  A chain's positions may be read in phases: phase 0 for every
// request, later ones for the requests whose drafts were all accepted so far.
struct Phase {
    int p0;                   // first node (position) of the phase
    int t_rows, R;            // target rows p0 .. p0+t_rows-1, then draft rows p0 .. p0+R-t_rows-1 of a request
    int units, U;             // units of a row, items of a unit
    const int* undecided;     // null: every request; else [B], < 0: the request takes part
    float2* part;             // [B, R, units] partials of the rows' units
    unsigned* ticket;         // a later phase's unit counter, 0 at its start
};

struct StatsParams {
    const void* target;       // [B, n, V]
    const void* draft;        // [B, d_rows, V] (null when greedy)
    const int32_t* parents;   // tree [B, n] (null for the chain)
    int B, V, n, d_rows;
    int I;                    // 4 KB items per row
    float c_hi, c_lo;         // log2(e) / T as a float pair
    Phase ph;
    // a later phase: for the requests that the phase before decided (at a position in
    // [mass_lo, mass_hi)): the draw masses of the units of their row pair
    int mass_lo, mass_hi;
    const float4* stat;       // [B] statistics of the pair
    float* mass;              // [B, units]
    long long share, extra;   // phase 0: units of a warp, and how many warps take one more
    FastDiv by_units, by_R;
};

// ------------------------------------------------------------ small helpers
__device__ __forceinline__ uint4 ld_stream(const void* p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename T>
union Vec16 {
    uint4 q;
    T t[16 / sizeof(T)];
};

template <typename T>
__device__ __forceinline__ int misaligned_by(const T* row) {   // elements past a 16-byte boundary
    return (int)((reinterpret_cast<uintptr_t>(row) & 15u) / sizeof(T));
}

// Bytes [off, off + 16) of two vectors.
__device__ __forceinline__ uint4 shift16(const uint4& lo, const uint4& hi, int off) {
    uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    if (off & 8) {
#pragma unroll
        for (int i = 0; i < 6; ++i) w[i] = w[i + 2];
    }
    if (off & 4) {
#pragma unroll
        for (int i = 0; i < 5; ++i) w[i] = w[i + 1];
    }
    const int sh = (off & 3) * 8;
    return make_uint4(__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh),
                      __funnelshift_r(w[2], w[3], sh), __funnelshift_r(w[3], w[4], sh));
}

// row[start .. start + kPer) at any alignment; entries outside [0, V) read as
// -inf.  Vectors that lie inside the row come as two aligned ones shifted
// together (one when row + start is on a 16-byte boundary), the row's ends
// element by element.
template <typename T>
__device__ __forceinline__ uint4 load16_any(const T* row, int start, int V) {
    constexpr int kPer = 16 / (int)sizeof(T);
    const int off = (int)(reinterpret_cast<uintptr_t>(row + start) & 15u);   // bytes; the same in every lane
    const int a = start - off / (int)sizeof(T);
    if (a < 0 || a + (off ? 2 : 1) * kPer > V) {
        Vec16<T> v;
#pragma unroll
        for (int e = 0; e < kPer; ++e) v.t[e] = start + e >= 0 && start + e < V ? row[start + e] : (T)kNegInf;
        return v.q;
    }
    const uint4 lo = *reinterpret_cast<const uint4*>(row + a);
    return off ? shift16(lo, reinterpret_cast<const uint4*>(row + a)[1], off) : lo;
}

// count vectors, the u-th at start + u * step.  Not inlined: a kernel holds
// one copy of it for its row ends and odd rows, off the straight path (the
// latency of a short call is mostly instruction fetches).
template <typename T>
__device__ __noinline__ void load_slow(const T* row, int start, int step, int count, int V, uint4* out) {
#pragma unroll 1
    for (int u = 0; u < count; ++u) out[u] = load16_any(row, start + u * step, V);
}

// Whether the row's vectors lie wholly inside it or wholly past its end.
template <typename T>
__device__ __forceinline__ bool whole_vectors(const T* row, int V) {
    return ((reinterpret_cast<uintptr_t>(row) & 15u) | (unsigned)(V % (16 / (int)sizeof(T)))) == 0;
}

// The vector at start >= 0 of such a row.
template <typename T>
__device__ __forceinline__ uint4 load_or_ninf(const T* row, int start, int V) {
    Vec16<T> v;
#pragma unroll
    for (int e = 0; e < 16 / (int)sizeof(T); ++e) v.t[e] = (T)kNegInf;
    if (start < V) v.q = ld_stream(row + start);
    return v.q;
}

// Block j of a row (kN vectors per lane) into registers: lane l holds the
// vectors u * 32 + l.  The blocks of a row start at the 16-byte boundary at
// or before its first element, so rows of any alignment take vector loads.
template <typename T, int kN>
__device__ __forceinline__ void load_block(const T* row, int j, int V, int lane, uint4 (&v)[kN]) {
    constexpr int kPer = 16 / (int)sizeof(T);
    constexpr int kBlock = 32 * kN * kPer;
    const int base = j * kBlock - misaligned_by(row);
    if (base >= 0 && base + kBlock <= V) {
#pragma unroll
        for (int u = 0; u < kN; ++u) v[u] = ld_stream(row + base + (u * 32 + lane) * kPer);
    } else if (whole_vectors(row, V)) {
        // the last block of the usual row: its loads in flight together too
        // (one after the other: 8 requests, k = 5, V = 128256 14.0 us a call, 12.4
        // so; 256 requests, k = 8 142 and 133)
#pragma unroll
        for (int u = 0; u < kN; ++u) v[u] = load_or_ninf(row, base + (u * 32 + lane) * kPer, V);
    } else {
        uint4 t[kN];
        load_slow(row, base + lane * kPer, 32 * kPer, kN, V, t);
#pragma unroll
        for (int u = 0; u < kN; ++u) v[u] = t[u];
    }
}

// kN vectors of a row pair, the u-th at first + u * step, on the target row's
// 16-byte boundaries: base is the block's first element, size its elements.
// Where the draft row lies differently on those boundaries its vectors come as
// two aligned ones shifted together.  (Through the out-of-line routine, one
// after the other: 68 requests, k = 3, V = 65950, fp32 43.9 us a call, 36.3 so; 316,
// k = 3, V = 90074, bf16 150 and 115.)
template <typename T, int kN>
__device__ __forceinline__ void load_pair(const T* rt, const T* rd, bool same, int base, int size, int first, int step,
                                          int V, uint4 (&t)[kN], uint4 (&d)[kN]) {
    constexpr int kPer = 16 / (int)sizeof(T);
    if (base >= 0 && base + size <= V && same) {
#pragma unroll
        for (int u = 0; u < kN; ++u) {
            t[u] = *reinterpret_cast<const uint4*>(rt + first + u * step);
            d[u] = *reinterpret_cast<const uint4*>(rd + first + u * step);
        }
    } else if (same && whole_vectors(rt, V)) {
#pragma unroll
        for (int u = 0; u < kN; ++u) {
            t[u] = load_or_ninf(rt, first + u * step, V);
            d[u] = load_or_ninf(rd, first + u * step, V);
        }
    } else if (!same && base >= kPer && base + size + kPer <= V) {
        const int off = (int)(reinterpret_cast<uintptr_t>(rd + first) & 15u);   // bytes, not 0; the same in every lane
        const uint4* const q = reinterpret_cast<const uint4*>(rd + first - off / (int)sizeof(T));
        uint4 hi[kN];
#pragma unroll
        for (int u = 0; u < kN; ++u) {
            t[u] = *reinterpret_cast<const uint4*>(rt + first + u * step);
            d[u] = q[u * step / kPer];
            hi[u] = q[u * step / kPer + 1];
        }
#pragma unroll
        for (int u = 0; u < kN; ++u) d[u] = shift16(d[u], hi[u], off);
    } else {
        uint4 x[2 * kN];
        load_slow(rt, first, step, kN, V, x);
        load_slow(rd, first, step, kN, V, x + kN);
#pragma unroll
        for (int u = 0; u < kN; ++u) {
            t[u] = x[u];
            d[u] = x[kN + u];
        }
    }
}

// A pair (m, s) stands for sum_v 2^((z_v - m) c); empty is (-inf, 0).
__device__ __forceinline__ void fold(float& m, float& s, float m2, float s2, float c_hi, float c_lo) {
    const float M = fmaxf(m, m2);
    if (M == kNegInf) return;
    const float a = m == kNegInf ? 0.f : s * ex2_scaled(m - M, c_hi, c_lo);
    const float b = m2 == kNegInf ? 0.f : s2 * ex2_scaled(m2 - M, c_hi, c_lo);
    s = a + b;
    m = M;
}

// (max, id) with the lowest id on ties; the id travels as int bits.
__device__ __forceinline__ void argmax_fold(float2& acc, float2 o) {
    if (o.x > acc.x || (o.x == acc.x && __float_as_int(o.y) < __float_as_int(acc.y))) acc = o;
}

__device__ __forceinline__ float warp_incl_scan(float x, int lane) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    return x;
}

__device__ __forceinline__ int warp_max_int(int x) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, off));
    return x;
}

// Folds the (m, s) pairs of the 32 lanes: the maximum first, then one
// rescale per lane and a butterfly sum.  Every lane ends with the same pair.
__device__ __forceinline__ float2 warp_fold_sum(float m, float s, float c_hi, float c_lo) {
    float M = m;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
    float t = m == kNegInf ? 0.f : s * ex2_scaled(m - M, c_hi, c_lo);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    return make_float2(M, t);
}

// (max, lowest id of the max) over the 32 lanes, in every lane.
__device__ __forceinline__ float2 warp_fold_argmax(float2 acc) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        float2 o;
        o.x = __shfl_xor_sync(0xffffffffu, acc.x, off);
        o.y = __shfl_xor_sync(0xffffffffu, acc.y, off);
        argmax_fold(acc, o);
    }
    return acc;
}

// Bit u set iff tree node u of the parent array `par` (n <= 64 nodes) has a
// child; every lane of the warp returns the same mask.
__device__ __forceinline__ uint64_t tree_child_mask(const int32_t* par, int n, int lane) {
    uint64_t m = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        if (c > 0 && c < n) {
            const int q = par[c];
            if (q >= 0 && q < c) m |= 1ull << q;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m |= __shfl_xor_sync(0xffffffffu, m, off);
    return m;
}

// Out of line: a phase's start has four of them.
__device__ __noinline__ long long div_nn(long long x, long long d) { return div_pos(x, d); }

// ------------------------------------------------------------ kernel 1
// Largest of the logits of one lane's vectors (bf16: packed maxima, one
// instruction per pair).
template <int kN>
__device__ __forceinline__ float item_max(const uint4 (&v)[kN], __nv_bfloat16) {
    __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&v[0].x);
    __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&v[0].y);
    __nv_bfloat162 c = *reinterpret_cast<const __nv_bfloat162*>(&v[0].z);
    __nv_bfloat162 d = *reinterpret_cast<const __nv_bfloat162*>(&v[0].w);
#pragma unroll
    for (int u = 1; u < kN; ++u) {
        a = __hmax2(a, *reinterpret_cast<const __nv_bfloat162*>(&v[u].x));
        b = __hmax2(b, *reinterpret_cast<const __nv_bfloat162*>(&v[u].y));
        c = __hmax2(c, *reinterpret_cast<const __nv_bfloat162*>(&v[u].z));
        d = __hmax2(d, *reinterpret_cast<const __nv_bfloat162*>(&v[u].w));
    }
    a = __hmax2(__hmax2(a, b), __hmax2(c, d));
    return fmaxf(__low2float(a), __high2float(a));
}

template <int kN>
__device__ __forceinline__ float item_max(const uint4 (&v)[kN], float) {
    float a = kNegInf, b = kNegInf;
#pragma unroll
    for (int u = 0; u < kN; ++u) {
        a = fmaxf(a, fmaxf(__uint_as_float(v[u].x), __uint_as_float(v[u].y)));
        b = fmaxf(b, fmaxf(__uint_as_float(v[u].z), __uint_as_float(v[u].w)));
    }
    return fmaxf(a, b);
}

// The logits of a vector as fp32 pairs.
__device__ __forceinline__ void to_pairs(const uint4& v, uint64_t (&z)[4], __nv_bfloat16) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i] = f2_pack(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
}
__device__ __forceinline__ void to_pairs(const uint4& v, uint64_t (&z)[2], float) {
    z[0] = f2_pack(__uint_as_float(v.x), __uint_as_float(v.y));
    z[1] = f2_pack(__uint_as_float(v.z), __uint_as_float(v.w));
}

// The weights 2^((z - m) c_hi) of a pair: subtraction and product rounded one
// after the other, in packed arithmetic (half the instructions of the scalar
// form, bit for bit its results).
__device__ __forceinline__ uint64_t weight2(uint64_t z, uint64_t m2, uint64_t c2) {
    float a, b;
    f2_unpack(f2_mul(f2_sub(z, m2), c2), a, b);
    return f2_pack(ex2(a), ex2(b));
}

// sum over one lane's vectors of 2^((z - m) c_hi), four independent partial sums.
template <typename T, int kN>
__device__ __forceinline__ float item_sum(const uint4 (&v)[kN], float m, float c_hi) {
    constexpr int kPairs = 8 / (int)sizeof(T);
    const uint64_t m2 = f2_pack(m, m), c2 = f2_pack(c_hi, c_hi);
    uint64_t s2[2] = {0ull, 0ull};   // +0.0f pairs
#pragma unroll
    for (int u = 0; u < kN; ++u) {
        uint64_t z[kPairs];
        to_pairs(v[u], z, T());
#pragma unroll
        for (int i = 0; i < kPairs; ++i) s2[i & 1] = f2_add(s2[i & 1], weight2(z[i], m2, c2));
    }
    float a, b, e, f;
    f2_unpack(s2[0], a, b);
    f2_unpack(s2[1], e, f);
    return (a + b) + (e + f);
}

// Greedy: one lane's running (max, lowest id of it) over its item, whose
// vector u holds the logits at0 + u * 32 * kPer ...
template <typename T, int kN>
__device__ __forceinline__ void item_argmax(const uint4 (&cur)[kN], int at0, float& m, int& id) {
    constexpr int kPer = 16 / (int)sizeof(T);
#pragma unroll
    for (int u = 0; u < kN; ++u) {   // ascending ids: strict > keeps the lowest
        Vec16<T> v;
        v.q = cur[u];
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            const float z = to_f(v.t[e]);
            if (z > m) {
                m = z;
                id = at0 + u * 32 * kPer + e;
            }
        }
    }
}

// The draw weights are p and max(p - kappa q, 0) scaled by S_t (the inverse
// CDF does not depend on a common factor): 2^((zt - mt)c) and
// max(2^((zt - mt)c) - rho 2^((zd - md)c), 0) with rho = kappa S_t / S_d.
// p alone is rho = 0 with the target row in both places.
template <typename T>
struct DrawRow {
    const T* rt;
    const T* rd;
    float mt, md, rho, c_hi;
    bool same;   // both rows lie alike on 16-byte boundaries
};

// The pair's weights from its rows' statistics (a row without a finite entry,
// outside the contract, weighs zero everywhere); kappa == 0: p alone.
template <typename T>
__device__ __forceinline__ void set_weights(DrawRow<T>& d, float2 st, float2 sd, float kappa, float c_hi) {
    d.c_hi = c_hi;
    d.mt = st.x == kNegInf ? 0.f : st.x;
    d.md = sd.x == kNegInf ? 0.f : sd.x;
    d.rho = sd.y > 0.f ? kappa * (st.y / sd.y) : 0.f;
    if (!(kappa > 0.f)) {
        d.rd = d.rt;
        d.md = d.mt;
        d.rho = 0.f;
    }
    d.same = misaligned_by(d.rt) == misaligned_by(d.rd);
}

// The weights of a vector of both rows.
template <typename T>
__device__ __forceinline__ void weigh(const DrawRow<T>& d, const uint4& t, const uint4& q, float* w) {
    constexpr int kPairs = 8 / (int)sizeof(T);
    const uint64_t mt = f2_pack(d.mt, d.mt), md = f2_pack(d.md, d.md), c2 = f2_pack(d.c_hi, d.c_hi);
    const uint64_t nr = f2_pack(-d.rho, -d.rho);
    uint64_t zt[kPairs], zd[kPairs];
    to_pairs(t, zt, T());
    to_pairs(q, zd, T());
#pragma unroll
    for (int i = 0; i < kPairs; ++i) {
        float a, b;
        f2_unpack(f2_fma(nr, weight2(zd[i], md, c2), weight2(zt[i], mt, c2)), a, b);
        w[2 * i] = fmaxf(a, 0.f);
        w[2 * i + 1] = fmaxf(b, 0.f);
    }
}

// Draw mass of items [i0, i1) of the target row's items, by one warp: half an
// item of both rows is in flight while the other half is summed.
template <typename T>
__device__ __forceinline__ float item_masses(const DrawRow<T>& d, int i0, int i1, int V, int lane) {
    constexpr int kPer = 16 / (int)sizeof(T), kN = kVecs / 2, kHalf = 32 * kN * kPer;
    const int mis = misaligned_by(d.rt);
    auto load = [&](int h, uint4 (&t)[kN], uint4 (&q)[kN]) {
        const int base = h * kHalf - mis;
        load_pair(d.rt, d.rd, d.same, base, kHalf, base + lane * kPer, 32 * kPer, V, t, q);
    };
    auto sum = [&](const uint4 (&t)[kN], const uint4 (&q)[kN]) {
        float acc = 0.f;
#pragma unroll
        for (int u = 0; u < kN; ++u) {
            float w[kPer];
            weigh(d, t[u], q[u], w);
            float s = 0.f;
#pragma unroll
            for (int e = 0; e < kPer; ++e) s += w[e];
            acc += s;
        }
        return acc;
    };
    uint4 ta[kN], qa[kN], tb[kN], qb[kN];
    float acc = 0.f;
    load(2 * i0, ta, qa);
#pragma unroll 1
    for (int i = i0; i < i1; ++i) {
        load(2 * i + 1, tb, qb);
        acc += sum(ta, qa);
        if (i + 1 < i1) load(2 * i + 2, ta, qa);
        acc += sum(tb, qb);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    return acc;
}

// The grid fills the device once.  A unit is up to U items of one row and
// leaves one partial, so the results do not depend on which warp takes it.
// Phase 0 deals every warp an equal contiguous range of units.  kLater, the
// phases after it: the requests still undecided, and one row of draw masses
// for each that the phase before decided, are listed first; the last quarter
// of the units goes to whichever warp is free, by a counter (a short phase
// dealt out in equal shares ended 20-30% after its mean).  A warp keeps the next item in flight
// while it reduces the current one, across units.
// kShort, phase 0 of a call with few items a warp: one copy of the reduction,
// the items changing registers, where two copies in turn save that (7% of a
// long call): 16 requests, k = 5, V = 128256 22.3 us a call and 21.3 so, 8 from
// a flushed L2 24.8 and 24.3.
template <typename T, bool kGreedy, bool kLater, bool kShort>
__global__ void __launch_bounds__(kThreads, 2) accept_stats_kernel(const StatsParams p) {
    constexpr int kPer = 16 / (int)sizeof(T);
    constexpr int kItem = kItemBytes / (int)sizeof(T);
    constexpr bool kMass = kLater && !kGreedy;
    __shared__ uint16_t s_list[kLater ? kMaxPhased : 1];   // undecided requests from the front, decided from the back
    __shared__ int s_wcount[2][kWarps];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int I = p.I, V = p.V, R = p.ph.R, t_rows = p.ph.t_rows, p0 = p.ph.p0, units = p.ph.units, U = p.ph.U;
    const T* rp = nullptr;   // row, items and partial of the unit whose items are being loaded
    int item = 0, end = 0, at = 0;
    long long slot = 0;
    bool skip = false, drafted = false;
    auto open_unit = [&](long long x) {
        const long long row = p.by_units.div(x);
        const int u = (int)(x - row * units);
        const int idx = (int)p.by_R.div(row), r = (int)(row - (long long)idx * R);
        const int b = kLater ? s_list[idx] : idx;
        at = p0 + (r < t_rows ? r : r - t_rows);   // the row's node
        drafted = r >= t_rows;
        rp = !drafted ? static_cast<const T*>(p.target) + ((size_t)b * p.n + at) * V
                      : static_cast<const T*>(p.draft) + ((size_t)b * p.d_rows + at) * V;
        item = u * U;
        end = min(item + U, I);
        slot = ((long long)b * R + r) * units + u;
    };
    // tree: the draft row of a node without children is never used
    auto set_skip = [&]() {
        if (!kLater && !kGreedy && p.parents) {
            const int b = (int)p.by_R.div(p.by_units.div(slot));
            skip = drafted && !((tree_child_mask(p.parents + (size_t)b * p.n, p.n, lane) >> at) & 1ull);
        }
    };
    // phase 0 knows its shares before it reads anything, and works them out
    // before the wait, with no division (after it, with two: 15.0 us a call of
    // B = 8, k = 5, V = 128256, 14.2 so).  The warps with one unit more are
    // spread over the CTAs.
    long long unit = 0, hi = 0;
    if (!kLater) {
        const long long w = (long long)wid * gridDim.x + blockIdx.x;
        unit = w * p.share + min(w, p.extra);
        hi = unit + p.share + (w < p.extra ? 1 : 0);
        if (unit < hi) open_unit(unit);
    }
    // launched as a programmatic dependent of the kernel before it: its
    // inputs are read only past this wait, and the next kernel (which
    // reads some inputs before its own wait) only starts after it
    wait_prior_grid();
    allow_dependent_launch();
    int requests = p.B, massed = 0;
    if (kLater) {
        requests = 0;
        for (int b0 = 0; b0 < p.B; b0 += kThreads) {
            const int a = b0 + tid < p.B ? __ldcg(p.ph.undecided + b0 + tid) : INT_MAX;
            const bool in = a < 0, mass = kMass && a >= p.mass_lo && a < p.mass_hi;
            const unsigned m0 = __ballot_sync(0xffffffffu, in), m1 = __ballot_sync(0xffffffffu, mass);
            if (lane == 0) {
                s_wcount[0][wid] = __popc(m0);
                s_wcount[1][wid] = __popc(m1);
            }
            __syncthreads();
            int at0 = requests + __popc(m0 & ((1u << lane) - 1u)), at1 = massed + __popc(m1 & ((1u << lane) - 1u));
#pragma unroll 1
            for (int i = 0; i < kWarps; ++i) {
                const int n0 = s_wcount[0][i], n1 = s_wcount[1][i];
                if (i < wid) {
                    at0 += n0;
                    at1 += n1;
                }
                requests += n0;
                massed += n1;
            }
            if (in) s_list[at0] = (uint16_t)(b0 + tid);
            if (mass) s_list[kMaxPhased - 1 - at1] = (uint16_t)(b0 + tid);
            __syncthreads();
        }
    }
    // contiguous shares; of a later phase the last quarter goes by the counter
    const int W = (int)gridDim.x * kWarps, w = (int)blockIdx.x * kWarps + wid;
    const long long N = (long long)requests * R * units, fixed = N - N / 4;
    if (kLater) {
        unit = div_nn(w * fixed, W);
        hi = div_nn((w + 1) * fixed, W);
    }
    // One item into registers: lane l holds vectors u*32 + l; entries past
    // the row's end, and skipped rows, read as -inf.
    auto load = [&](uint4 (&v)[kVecs]) {
        if (skip) {
            Vec16<T> ninf;
#pragma unroll
            for (int e = 0; e < 16 / (int)sizeof(T); ++e) ninf.t[e] = (T)kNegInf;
#pragma unroll
            for (int u = 0; u < kVecs; ++u) v[u] = ninf.q;
            return;
        }
        load_block(rp, item, V, lane, v);
    };

    if (kMass) {
        // draw masses first: their rows were read last, so they are in L2
        const long long M = (long long)massed * units, m1 = div_nn((w + 1) * M, W);
#pragma unroll 1
        for (long long x = div_nn(w * M, W); x < m1; ++x) {
            const long long i = p.by_units.div(x);
            const int u = (int)(x - i * units), b = s_list[kMaxPhased - 1 - (int)i];
            const int a = __ldcg(p.ph.undecided + b);
            const float4 st = __ldcg(p.stat + b);
            DrawRow<T> d;
            d.rt = static_cast<const T*>(p.target) + ((size_t)b * p.n + a) * V;
            d.rd = static_cast<const T*>(p.draft) + ((size_t)b * p.d_rows + a) * V;
            set_weights(d, make_float2(st.x, st.y), make_float2(st.z, st.w), 1.f, p.c_hi);
            const float acc = item_masses(d, u * U, min((u + 1) * U, I), V, lane);
            if (lane == 0) p.mass[(size_t)b * units + u] = acc;
        }
    }
    if (N == 0) return;
    unsigned next = 0;   // the ticket taken ahead (lane 0)
    if (kLater && unit + 1 >= hi && lane == 0) next = atomicAdd(p.ph.ticket, 1u);
    if (unit >= hi) {
        if (!kLater) return;
        unit = fixed + __shfl_sync(0xffffffffu, next, 0);
        if (unit >= N) return;
        if (lane == 0) next = atomicAdd(p.ph.ticket, 1u);
    }
    if (kLater) open_unit(unit);
    else set_skip();

    float m = kNegInf, s = 0.f;            // sampling: lane's running (max, sum)
    int id = INT_MAX;                      // greedy: lane's lowest id of the max (m)
    bool more = true;
    // reduces the item in `cur` while the next one lands in `nxt`
    auto step = [&](uint4 (&cur)[kVecs], uint4 (&nxt)[kVecs]) {
        const int at0 = kGreedy ? item * kItem - misaligned_by(rp) + lane * kPer : 0;
        const long long done = slot;
        const bool unit_end = ++item == end;
        if (unit_end) {
            ++unit;
            if (kLater && unit >= hi) {
                unit = fixed + __shfl_sync(0xffffffffu, next, 0);
                more = unit < N;
            } else {
                more = unit < hi;
            }
            if (more) {
                open_unit(unit);
                set_skip();
            }
        }
        if (more) load(nxt);
        // a ticket ahead from the share's last unit on
        if (kLater && unit_end && more && unit + 1 >= hi && lane == 0) next = atomicAdd(p.ph.ticket, 1u);
        if (kGreedy) {
            item_argmax<T>(cur, at0, m, id);
        } else {
            const float mi = item_max(cur, T());
            if (mi > m) {
                s = m == kNegInf ? 0.f : s * ex2_scaled(m - mi, p.c_hi, p.c_lo);
                m = mi;
            }
            if (m != kNegInf) s += item_sum<T>(cur, m, p.c_hi);
        }
        if (unit_end) {
            // fold the lanes and publish the pair
            const float2 acc = kGreedy ? warp_fold_argmax(make_float2(m, __int_as_float(id)))
                                       : warp_fold_sum(m, s, p.c_hi, p.c_lo);
            if (lane == 0) p.ph.part[done] = acc;
            m = kNegInf;
            s = 0.f;
            id = INT_MAX;
        }
    };
    uint4 va[kVecs], vb[kVecs];
    load(va);
    for (;;) {
        step(va, vb);
        if (!more) break;
        if (kShort) {
#pragma unroll
            for (int u = 0; u < kVecs; ++u) va[u] = vb[u];
        } else {
            step(vb, va);
            if (!more) break;
        }
    }
}

// Statistics of kBatch rows (r0, r0 + step, ... below R) of request b: lane l
// folds units l, l + 32, ... in order, then the lanes; the same numbers in
// every warp that folds the row.  The rows' loads are in flight together.
template <bool kGreedy, int kBatch>
__device__ __forceinline__ void fold_rows(const Phase& ph, int b, int r0, int step, int lane, float c_hi, float c_lo,
                                          float2 (&f)[kBatch]) {
    const float2 empty = make_float2(kNegInf, kGreedy ? __int_as_float(INT_MAX) : 0.f);
    const float2* const part = ph.part + (size_t)b * ph.R * ph.units;
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
        const int r = r0 + i * step;
        f[i] = r < ph.R && lane < ph.units ? __ldcg(part + (size_t)r * ph.units + lane) : empty;
    }
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
        const int r = r0 + i * step;
#pragma unroll 1
        for (int l = lane + 32; r < ph.R && l < ph.units; l += 32) {
            const float2 o = __ldcg(part + (size_t)r * ph.units + l);
            if (kGreedy) argmax_fold(f[i], o);
            else fold(f[i].x, f[i].y, o.x, o.y, c_hi, c_lo);
        }
        f[i] = kGreedy ? warp_fold_argmax(f[i]) : warp_fold_sum(f[i].x, f[i].y, c_hi, c_lo);
    }
}

// ------------------------------------------------------------ accept test
// p(x) / q(x) of a drafted token: zt, zd are its target and draft logits,
// st, sd the rows' statistics; 0 for an invalid token or p(x) == 0, +inf
// when q(x) == 0.
__device__ __forceinline__ float accept_ratio(bool valid, float zt, float zd, float2 st, float2 sd,
                                              float c_hi, float c_lo) {
    if (!valid || zt == kNegInf) return 0.f;
    if (zd == kNegInf) return __int_as_float(0x7f800000);
    // log2 p(x)/q(x) = ((zt - mt) - (zd - md)) c + log2 Sd - log2 St, carried
    // as an unevaluated float pair
    const float dz = (zt - st.x) - (zd - sd.x);
    const float A = dz * c_hi;
    float E = fmaf(dz, c_lo, fmaf(dz, c_hi, -A));
    const float Bl = lg2(sd.y) - lg2(st.y);
    const float H = A + Bl;
    const float bb = H - A;
    E += (A - (H - bb)) + (Bl - bb);
    return ex2(H) * fmaf(E, kLn2, 1.f);
}

// ------------------------------------------------------------ test kernel
// What a phase decides: per request the accepted count a, or -1 while every
// position so far is accepted, and the statistics of the deciding row pair
// (greedy: the emitted token's bits in x).
struct Decided {
    int* a;        // [B]
    float4* stat;  // [B]
};

struct TestParams {
    const void* target;
    const void* draft;
    const int32_t* tokens;    // [B, n-1]
    const float* uniforms;    // [B, n]
    int B, V, n;
    float c_hi, c_lo;
    Phase ph;
    Decided dec;
};

// One warp per request tests the positions of a phase (a single phase's are
// tested by the walk kernel).
template <typename T, bool kGreedy>
__global__ void __launch_bounds__(kThreads) accept_test_kernel(const TestParams p) {
    constexpr int kBatch = 4;
    __shared__ float2 s_stat[kWarps][2 * kMaxTreeNodes];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int b = blockIdx.x * kWarps + wid;
    const int p0 = p.ph.p0, g = p.ph.t_rows, R = p.ph.R;
    const int tests = min(g, p.n - 1 - p0);   // positions with a draft (all but a chain's last)
    int x = -1;
    float zt = kNegInf, zd = 0.f, u = 1.f;
    if (b < p.B && lane < tests) {
        x = p.tokens[(size_t)b * (p.n - 1) + p0 + lane];
        if (!kGreedy) {
            u = p.uniforms[(size_t)b * p.n + p0 + lane];
            if (x >= 0 && x < p.V) {
                zt = to_f(static_cast<const T*>(p.target)[((size_t)b * p.n + p0 + lane) * p.V + x]);
                zd = to_f(static_cast<const T*>(p.draft)[((size_t)b * (p.n - 1) + p0 + lane) * p.V + x]);
            }
        }
    }
    wait_prior_grid();
    allow_dependent_launch();
    if (blockIdx.x == 0 && threadIdx.x == 0) *p.ph.ticket = 0;   // for the next phase
    if (b >= p.B) return;
    if (p.ph.undecided && __ldcg(p.ph.undecided + b) >= 0) return;
#pragma unroll 1
    for (int r0 = 0; r0 < R; r0 += kBatch) {
        float2 f[kBatch];
        fold_rows<kGreedy, kBatch>(p.ph, b, r0, 1, lane, p.c_hi, p.c_lo, f);
#pragma unroll
        for (int i = 0; i < kBatch; ++i)
            if (lane == i && r0 + i < R) s_stat[wid][r0 + i] = f[i];
    }
    __syncwarp();
    bool rej = false;
    int top = 0;
    float2 st = make_float2(0.f, 0.f), sd = st;
    if (lane < g) {
        st = s_stat[wid][lane];
        if (kGreedy) {
            top = __float_as_int(st.y);
            if (top == INT_MAX) top = 0;   // a row with no finite entry
            rej = lane < tests && x != top;
        } else if (lane < tests) {
            sd = s_stat[wid][g + lane];
            rej = !(u < accept_ratio(zt != kNegInf, zt, zd, st, sd, p.c_hi, p.c_lo));
        }
    }
    const unsigned m = __ballot_sync(0xffffffffu, rej);
    const int at = m ? __ffs(m) - 1 : tests;   // the deciding position
    if (at == g) {
        if (lane == 0) p.dec.a[b] = -1;
    } else if (lane == at) {
        p.dec.a[b] = p0 + lane;
        p.dec.stat[b] = kGreedy ? make_float4(__int_as_float(top), 0.f, 0.f, 0.f) : make_float4(st.x, st.y, sd.x, sd.y);
    }
}

// ------------------------------------------------------------ cluster PTX
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}

__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

#include "spec_accept_walk.cuh"

// ------------------------------------------------------------------- host
std::atomic<int> g_max_cluster[64];

// The largest cluster (16, non-portable, or 8) the device schedules for the
// walk kernel.
int max_cluster_size() {
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 8;
    if (g_max_cluster[dev]) return g_max_cluster[dev];
    int best = 8;
    const void* kerns[8] = {(const void*)accept_walk_kernel<__nv_bfloat16, false, false>,
                            (const void*)accept_walk_kernel<float, false, false>,
                            (const void*)accept_walk_kernel<__nv_bfloat16, true, false>,
                            (const void*)accept_walk_kernel<float, true, false>,
                            (const void*)accept_walk_kernel<__nv_bfloat16, false, true>,
                            (const void*)accept_walk_kernel<float, false, true>,
                            (const void*)accept_walk_kernel<__nv_bfloat16, true, true>,
                            (const void*)accept_walk_kernel<float, true, true>};
    bool attrs_ok = true;
    for (auto k : kerns)
        attrs_ok = attrs_ok && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    if (attrs_ok) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kMaxCluster, 1, 1);
        cfg.blockDim = dim3(kWalkMaxThreads, 1, 1);
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = kMaxCluster;
        attr.val.clusterDim.y = 1;
        attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        bool all = true;
        for (auto k : kerns) {
            int n = 0;
            all = all && cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n > 0;
        }
        if (all) best = kMaxCluster;
    }
    cudaGetLastError();
    g_max_cluster[dev] = best;
    return best;
}

constexpr int kMaxPhases = 4;

struct AcceptPlan {
    int I;                                     // items of a row
    int phases, start[kMaxPhases + 1];         // nodes [start[i], start[i+1]) are read in phase i (0: the walk streams)
    int units, U;                              // units of a row, items of a unit
    int cluster, threads, blocks, per;   // the walk
    size_t off_mass, off_stat, off_a, off_ticket, bytes;
};

// n nodes per request (chain: k + 1; tree), on rows at 16-byte boundaries or not.
AcceptPlan plan_accept(const cs_accept_dims& d, int n, bool tree, bool greedy, bool aligned) {
    const bool f32 = d.logit_dtype == CS_F32;
    const int esz = f32 ? 4 : 2, item = kItemBytes / esz, sms = current_sm_count();
    AcceptPlan P{};
    P.I = (int)(((long long)d.vocab + (aligned ? 0 : 16 / esz - 1) + item - 1) / item);
    // The cluster: the CTAs of all requests in one wave (two an SM), a power
    // of two (they pack a GPC; nine CTAs a request took 40 us where eight took
    // 35, B = 32).
    int c = 1;
    while (2 * c <= max_cluster_size() && 2ll * c * d.batch <= 2 * sms) c *= 2;
    // one position of every request, in us at the copy bandwidth
    const double pos_us = (double)d.batch * d.vocab * esz * (greedy || n == 1 ? 1 : 2) / 6.5e6;
    // A tree whose nodes' rows take longer than a few rounds of the walk is
    // streamed by it: 34 nodes, V = 128256, bf16: 31 us (B = 8), against 50
    // when every row is read first; 7 nodes in a chain: 35 against 17.
    const bool stream = tree && n * pos_us >= 8.0;
    if (!stream) {
        // The first phase takes the positions of about 30 us, every later one
        // twice as many as were read before it, and what is left over when it
        // is less than 15 us joins the last; 7.5 us are enough for the first
        // split of a sampled call, which also takes the weighing from the walk
        // (B = 256, k = 2, V = 128256, bf16 at once 75 to 86 us, in two phases 71 to
        // 78; B = 160, fp32 99 to 116 and 82 to 91).
        // The first split costs about 15 us (a test, hand-offs, an uneven end, the
        // last masses), a further one 6, and a call whose drafts are nearly all
        // accepted gets nothing for them.  So a call is read in phases where that
        // loses next to nothing (us with 0.95, 0.8 and 0.6 of the drafts accepted,
        // V = 128256, bf16):
        //  - a greedy call from 60 us on (it has no masses): B = 256, k = 8 92 and
        //    56 with 0.95 and 0.7 accepted, in three phases 94 and 59, at once 92 and 92;
        //  - a sampled one from 60 us on where the walk would otherwise weigh more
        //    than 350 KB of a row pair in one CTA, which takes about as long as a
        //    split: B = 256, k = 3 94, 94, 94, at once 95, 101, 105 (B = 64, k = 5,
        //    V = 151936, fp32, 304 KB: 91 with 0.95, at once 78);
        //  - any other from 100 us on: B = 128, k = 8 (91 us) 115, 99, 89, at once
        //    100, 104, 106; k = 11 (121 us) in two phases 134, 112, 92, at once 127,
        //    132, 133;
        //  - in two phases up to 150 us, then in as many as there are: k = 11 in three
        //    137, 108, 92; B = 128, k = 16 (172 us) in four 180, 125, 99, in two 176,
        //    134, 99, at once 175, 180, 181; B = 256, k = 8 (182 us) in three 187, 158,
        //    127, in two 184, 169, 143, at once 191, 200, 202.
        // fp32 rows of the same bytes lie within 8% of these: B = 64, k = 8 (91 us)
        // 109, 98, 90, at once 93, 99, 101; B = 64, k = 16 (172 us) 174, 127, 93, at once
        // 166, 172, 172.
        constexpr double kPhaseUs = 30.0, kShareBytes = 350e3;
        const double call_us = n * pos_us;
        const bool pays = greedy || 2.0 * d.vocab * esz / c > kShareBytes;
        const int most = tree || d.batch > kMaxPhased || call_us < (pays ? 60.0 : 100.0) ? 1
                         : call_us < 150.0 ? 2 : kMaxPhases;
        P.phases = 1;
        long long g = most > 1 ? (long long)(kPhaseUs / pos_us) + 1 : n;
        // (the last position has no draft row)
        while (P.phases < most && g < n &&
               (n - g - (greedy ? 0.0 : 0.5)) * pos_us >= (P.phases == 1 && !greedy ? kPhaseUs / 4 : kPhaseUs / 2)) {
            P.start[P.phases++] = (int)g;
            g *= 2;
        }
        P.start[P.phases] = n;
    }
    // A streamed tree's cluster has at least four CTAs, for its rounds' latency.
    // Decided requests, the sampler and greedy calls have no slices to share.
    P.threads = kWalkMaxThreads;
    if (stream) {
        if (c < 4) c = 4;
    } else if (P.phases > 1 || greedy || n == 1) {
        c = 1;
        if (n > 1) P.threads = 64;
    }
    // A long row takes more CTAs, 512 blocks each; where the device has no
    // cluster of that many, the largest one holds up to twice that a CTA.
    constexpr int kRowBlocks = 512, kMostBlocks = kWalkSegs * kRunVecs / kWalkVecs;
    static_assert((CS_MAX_VOCAB * 4ll + 12 + kWalkVecs * 512 - 1) / (kWalkVecs * 512) <= 8 * kMostBlocks,
                  "a portable cluster holds the longest row, at any alignment");
    const int block = 32 * kWalkVecs * 16 / esz;
    P.blocks = (int)(((long long)d.vocab + (aligned ? 0 : 16 / esz - 1) + block - 1) / block);
    int need = (P.blocks + kRowBlocks - 1) / kRowBlocks;
    if (need > max_cluster_size()) need = max_cluster_size();
    if (c < need) c = need;
    if (c > P.blocks) c = P.blocks;
    P.cluster = c;
    P.per = (P.blocks + c - 1) / c;
    if (!stream && !greedy)
        while (P.threads > 64 && P.threads / 64 >= P.per && (long long)d.batch * c > sms) P.threads /= 2;   // tiny rows
    P.bytes = 256;
    if (P.phases > 0) {
        int g = 0;
        for (int i = 0; i < P.phases; ++i)
            if (P.start[i + 1] - P.start[i] > g) g = P.start[i + 1] - P.start[i];
        const size_t rows = (size_t)d.batch * (greedy ? g : 2 * g);
        P.U = (long long)rows * P.I <= 2ll * kWarps * sms ? 1 : P.I <= 64 ? 2 : P.I <= 256 ? 4 : 8;
        P.units = (P.I + P.U - 1) / P.U;
        auto up = [](size_t x) { return (x + 255) / 256 * 256; };
        P.off_mass = up(rows * P.units * sizeof(float2));
        P.off_stat = P.off_mass + (P.phases > 1 && !greedy ? up((size_t)d.batch * P.units * sizeof(float)) : 0);
        P.off_a = P.off_stat + up(d.batch * sizeof(float4));
        P.off_ticket = P.off_a + up(d.batch * sizeof(int));
        P.bytes = P.off_ticket + 256;
    }
    return P;
}

// The scratch of a call, wherever its rows lie.
size_t workspace_bytes(const cs_accept_dims& d, int n, bool tree, bool greedy) {
    const size_t a = plan_accept(d, n, tree, greedy, true).bytes, b = plan_accept(d, n, tree, greedy, false).bytes;
    return a > b ? a : b;
}

// Every kernel of a call is a programmatic dependent of the kernel before it:
// it may start early and waits (griddepcontrol.wait) before it reads what
// that kernel wrote.
template <typename Kern, typename Params>
cudaError_t launch_after(Kern kern, unsigned gx, unsigned gy, int threads, int cluster, cudaStream_t stream,
                         const Params& p) {
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = 1;
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = cluster;
    attrs[1].val.clusterDim.y = 1;
    attrs[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(gx, gy, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.stream = stream;
    cfg.attrs = attrs;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, p);
}

template <typename T, bool G>
cs_status launch_typed(StatsParams sp, TestParams tp, WalkParams p, const AcceptPlan& P, bool tree, void* workspace,
                       cudaStream_t stream) {
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const Decided dec{reinterpret_cast<int*>(ws + P.off_a), reinterpret_cast<float4*>(ws + P.off_stat)};
    Phase ph{};
    ph.units = P.units;
    ph.U = P.U;
    ph.part = reinterpret_cast<float2*>(ws);
    ph.ticket = reinterpret_cast<unsigned*>(ws + P.off_ticket);
    sp.by_units.set(P.units);
    sp.stat = dec.stat;
    sp.mass = reinterpret_cast<float*>(ws + P.off_mass);
    const int fill = 2 * current_sm_count();   // two CTAs an SM (the kernel's launch bounds)
    for (int i = 0; i < P.phases; ++i) {
        const int g = P.start[i + 1] - P.start[i];
        const bool last = i + 1 == P.phases;
        ph.p0 = P.start[i];
        ph.t_rows = g;
        ph.R = G ? g : tree ? 2 * g : last ? 2 * g - 1 : 2 * g;
        ph.undecided = i ? dec.a : nullptr;
        sp.ph = ph;
        sp.mass_lo = i ? P.start[i - 1] : 0;
        sp.mass_hi = ph.p0;
        sp.by_R.set(ph.R);
        const long long ctas = ((long long)sp.B * ph.R * ph.units + kWarps - 1) / kWarps;
        const unsigned grid = (unsigned)(ctas < fill ? ctas : fill);
        sp.share = (long long)sp.B * ph.R * ph.units / ((long long)grid * kWarps);
        sp.extra = (long long)sp.B * ph.R * ph.units % ((long long)grid * kWarps);
        auto* const stats = i ? accept_stats_kernel<T, G, true, false>
                              : sp.share * ph.U < 8 ? accept_stats_kernel<T, G, false, true>
                                                    : accept_stats_kernel<T, G, false, false>;
        cudaError_t e = launch_after(stats, grid, 1, kThreads, 1, stream, sp);
        if (e != cudaSuccess) return cuda_fail(e, "accept_stats_kernel launch");
        if (P.phases == 1) break;
        tp.ph = ph;
        tp.dec = dec;
        e = launch_after(accept_test_kernel<T, G>, (unsigned)(sp.B + kWarps - 1) / kWarps, 1, kThreads, 1, stream, tp);
        if (e != cudaSuccess) return cuda_fail(e, "accept_test_kernel launch");
        if (last && !G && ph.p0 < sp.n - 1) {   // the masses of the pairs that the last phase decided
            sp.ph.p0 = sp.n;
            sp.ph.t_rows = sp.ph.R = 0;
            sp.ph.undecided = dec.a;
            sp.mass_lo = ph.p0;
            sp.mass_hi = sp.n - 1;
            sp.by_R.set(0);
            e = launch_after(accept_stats_kernel<T, G, true, false>, grid, 1, kThreads, 1, stream, sp);
            if (e != cudaSuccess) return cuda_fail(e, "accept_stats_kernel launch");
        }
    }
    if (P.phases > 1) ph.undecided = dec.a;
    p.mass = sp.mass;
    p.ph = ph;
    p.dec = dec;
    for (int b0 = 0; b0 < sp.B; b0 += 65535) {
        p.b_base = b0;
        const cudaError_t e = launch_after(P.phases ? accept_walk_kernel<T, G, false> : accept_walk_kernel<T, G, true>, P.cluster, sp.B - b0 < 65535 ? sp.B - b0 : 65535,
                                           P.threads, P.cluster, stream, p);
        if (e != cudaSuccess) return cuda_fail(e, "accept_walk_kernel launch");
    }
    return CS_OK;
}

cs_status launch_accept(const cs_accept_dims& d, const void* target, const void* draft, const int32_t* parents,
                        const int32_t* tokens, const float* uniforms, int n, float temperature, int32_t* out_tokens,
                        int32_t* out_path, int32_t* out_n, void* workspace, cudaStream_t stream) {
    const bool greedy = temperature == 0.f, tree = parents != nullptr;
    const size_t esz = d.logit_dtype == CS_F32 ? 4 : 2;
    const bool aligned = (size_t)d.vocab * esz % 16 == 0 &&
                         ((reinterpret_cast<uintptr_t>(target) | reinterpret_cast<uintptr_t>(draft)) & 15) == 0;
    const AcceptPlan P = plan_accept(d, n, tree, greedy, aligned);
    const double c = temperature > 0.f ? 1.4426950408889634 / (double)temperature : 0.0;
    StatsParams sp{};
    sp.target = target;
    sp.draft = draft;
    sp.parents = parents;
    sp.B = d.batch;
    sp.V = d.vocab;
    sp.n = n;
    sp.d_rows = tree ? n : n - 1;
    sp.I = P.I;
    sp.c_hi = (float)c;
    sp.c_lo = (float)(c - (double)sp.c_hi);
    TestParams tp{};
    tp.target = target;
    tp.draft = draft;
    tp.tokens = tokens;
    tp.uniforms = uniforms;
    tp.B = d.batch;
    tp.V = d.vocab;
    tp.n = n;
    tp.c_hi = sp.c_hi;
    tp.c_lo = sp.c_lo;
    WalkParams p{};
    p.target = target;
    p.draft = draft;
    p.tokens = tokens;
    p.uniforms = uniforms;
    p.parents = parents;
    p.out_tokens = out_tokens;
    p.out_n = out_n;
    p.out_path = out_path;
    p.B = d.batch;
    p.V = d.vocab;
    p.n = n;
    p.d_rows = sp.d_rows;
    p.I = P.I;
    p.blocks = P.blocks;
    p.per = P.per;
    p.c_hi = sp.c_hi;
    p.c_lo = sp.c_lo;
    if (d.logit_dtype == CS_F32)
        return greedy ? launch_typed<float, true>(sp, tp, p, P, tree, workspace, stream)
                      : launch_typed<float, false>(sp, tp, p, P, tree, workspace, stream);
    return greedy ? launch_typed<__nv_bfloat16, true>(sp, tp, p, P, tree, workspace, stream)
                  : launch_typed<__nv_bfloat16, false>(sp, tp, p, P, tree, workspace, stream);
}

}  // namespace

size_t accept_workspace_bytes(const cs_accept_dims& d, int n_draft, float temperature) {
    return workspace_bytes(d, n_draft + 1, false, temperature == 0.f);
}

size_t accept_workspace_bytes_any(const cs_accept_dims& d, int n_draft) {
    const size_t a = workspace_bytes(d, n_draft + 1, false, true);
    const size_t b = workspace_bytes(d, n_draft + 1, false, false);
    return a > b ? a : b;
}

cs_status launch_spec_accept(const cs_accept_dims& d, const void* target, const void* draft,
                             const int32_t* tokens, const float* uniforms, int n_draft,
                             float temperature, int32_t* out_tokens, int32_t* out_n,
                             void* workspace, cudaStream_t stream) {
    return launch_accept(d, target, draft, nullptr, tokens, uniforms, n_draft + 1, temperature, out_tokens, nullptr,
                         out_n, workspace, stream);
}

size_t tree_accept_workspace_bytes(const cs_accept_dims& d, int n_nodes) {
    const size_t a = workspace_bytes(d, n_nodes, true, true);
    const size_t b = workspace_bytes(d, n_nodes, true, false);
    return a > b ? a : b;
}

cs_status launch_tree_accept(const cs_accept_dims& d, const void* target, const void* draft,
                             const int32_t* parents, const int32_t* tokens, const float* uniforms, int n_nodes,
                             float temperature, int32_t* out_tokens, int32_t* out_path, int32_t* out_n,
                             void* workspace, cudaStream_t stream) {
    return launch_accept(d, target, draft, parents, tokens, uniforms, n_nodes, temperature, out_tokens, out_path,
                         out_n, workspace, stream);
}

}  // namespace cs
