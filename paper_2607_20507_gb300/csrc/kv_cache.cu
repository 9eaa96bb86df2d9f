// kv_cache.cu -- the paged KV cache around the verify pass: appending the
// K/V rows of the k+1 verify positions before verify attention, and
// committing the accepted prefix after the acceptance step (the target's
// draft-and-verify step, Sec. 3.4; the positions follow the convention of
// cs_verify_attention: ctx_lens counts the k+1 verify positions).
//
// Append: one thread moves 16 bytes; 16 threads move one 256-byte row of one
// head (D = 128 bf16), so every load of the new rows and every store into a
// page slot is a contiguous 256-byte segment.  Commit is one thread per
// request.
//
// All of these are small: what bounds them is the chain of dependent loads
// and the launch itself, so each starts as a programmatic dependent of the
// kernel before it (its CTAs are in place when that kernel's last CTA leaves)
// and reads what does not depend on another load at once.
//
// Tree commit (after a token-tree acceptance): the accepted nodes' rows move,
// in walk order, to the positions right after the root.  Node path[i] sat at
// L - n + path[i] >= L - n + 1 + i, so with the rows taken in ascending i no
// source is an earlier destination; the 16 threads of a (request, head,
// K or V) group each own one 16-byte column, so a destination that overwrites
// an earlier source is written by the thread that already read that source.
// One CTA per request: thread i looks up the pages of accepted node i, a
// column's rows are then read eight at a time before they are written, and
// the same CTA writes the kept length at the end.  (A path or table under
// which a row would be read after an earlier row was written over it is
// copied row after row.)
#include "cs_device.cuh"
#include "cs_internal.h"

namespace cs {
namespace {

constexpr int kAppendThreads = 256;
constexpr int kRowThreads = 16;   // 16 x 16 B = one 128-dim bf16 row

struct AppendParams {
    const uint4* new_k;        // [B, n_new, Hkv, D]
    const uint4* new_v;
    uint4* k_pages;            // [P, Hkv, ps, D]
    uint4* v_pages;
    const int32_t* page_table; // [B, max_pages]
    const int32_t* ctx_lens;   // [B]
    long long rows;            // B * n_new * Hkv
    int n_new, Hkv, ps, max_pages, P;
};

__global__ void __launch_bounds__(kAppendThreads) kv_append_kernel(const AppendParams p) {
    const long long t = (long long)blockIdx.x * kAppendThreads + threadIdx.x;
    const long long r = t / kRowThreads;   // (b, i, h) row of the new K/V
    const int c = (int)(t % kRowThreads);
    wait_prior_grid();
    allow_dependent_launch();
    if (r >= p.rows) return;
    const int h = (int)(r % p.Hkv);
    const long long bi = r / p.Hkv;
    const int i = (int)(bi % p.n_new);
    const int b = (int)(bi / p.n_new);
    const size_t src = (size_t)r * kRowThreads + c;
    int L = __ldcg(p.ctx_lens + b);
    const uint4 k = __ldcg(p.new_k + src), v = __ldcg(p.new_v + src);
    L = max(0, min(L, p.max_pages * p.ps));
    const int pos = L - p.n_new + i;          // key position of verify row i
    if (pos < 0) return;                      // the context cannot hold this row
    const int page = __ldcg(p.page_table + (size_t)b * p.max_pages + pos / p.ps);
    if (page < 0 || page >= p.P) return;      // no such page: nothing is written
    const size_t dst = (((size_t)page * p.Hkv + h) * p.ps + pos % p.ps) * kRowThreads + c;
    p.k_pages[dst] = k;
    p.v_pages[dst] = v;
}

__global__ void kv_commit_kernel(int32_t* ctx_lens, const int32_t* n_accepted, int batch, int n_draft) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    wait_prior_grid();
    allow_dependent_launch();
    if (b >= batch) return;
    // rows kept: the prefix, the verify input token and the accepted drafts
    const int L = __ldcg(ctx_lens + b) - n_draft + __ldcg(n_accepted + b);
    ctx_lens[b] = L > 0 ? L : 0;
}

constexpr int kCommitMaxThreads = 1024;
constexpr int kCommitRows = 8;    // rows of a column in flight

struct TreeCommitParams {
    uint4* k_pages;            // [P, Hkv, ps, D]
    uint4* v_pages;
    const int32_t* page_table; // [B, max_pages]
    int32_t* ctx_lens;         // [B]
    const int32_t* path;       // [B, n]
    const int32_t* n_accepted; // [B]
    int n, Hkv, ps, max_pages, P;
};

// One CTA per request of at least CS_MAX_TREE_NODES threads.
// Up to 8 accepted nodes are one round trip for the lengths and
// the path, one for the pages and one for the rows, where row after row took
// two for each node (8 requests, 34 nodes: 8.9 us with the length kernel apart,
// a step of it 104 us; 93 with this kernel and the early starts).
__global__ void __launch_bounds__(kCommitMaxThreads) kv_commit_tree_kernel(const TreeCommitParams p) {
    __shared__ long long s_src[CS_MAX_TREE_NODES], s_dst[CS_MAX_TREE_NODES];   // head 0's row, -1: not moved
    const int b = blockIdx.x, tid = threadIdx.x;
    wait_prior_grid();
    allow_dependent_launch();
    const int32_t* table = p.page_table + (size_t)b * p.max_pages;
    const int L = max(0, min(__ldcg(p.ctx_lens + b), p.max_pages * p.ps));
    const int a = max(0, min(__ldcg(p.n_accepted + b), p.n - 1));
    const int base = L - p.n;
    if (tid < p.n) {
        const int node = __ldcg(p.path + (size_t)b * p.n + tid);
        const int src = base + node, dst = base + 1 + tid;
        long long sr = -1, dr = -1;
        if (tid < a && node >= 1 && node < p.n && src != dst && src >= 0 && dst >= 0) {
            const int sp = __ldcg(table + src / p.ps), dp = __ldcg(table + dst / p.ps);
            if (sp >= 0 && sp < p.P && dp >= 0 && dp < p.P) {
                sr = (long long)sp * p.Hkv * p.ps + src % p.ps;
                dr = (long long)dp * p.Hkv * p.ps + dst % p.ps;
            }
        }
        s_src[tid] = sr;
        s_dst[tid] = dr;
    }
    __syncthreads();
    bool late = false;   // this row's source is written by an earlier row of its batch
    if (tid < a && s_src[tid] >= 0)
        for (int j = tid / kCommitRows * kCommitRows; j < tid; ++j) late |= s_dst[j] == s_src[tid];
    const int step = __syncthreads_or(late) ? 1 : kCommitRows;
    const long long columns = (long long)p.Hkv * 2 * kRowThreads;
    for (long long t = tid; t < columns; t += blockDim.x) {
        const int c = (int)(t % kRowThreads), h = (int)(t / (2 * kRowThreads));
        uint4* pool = ((t / kRowThreads) & 1 ? p.v_pages : p.k_pages) + (size_t)h * p.ps * kRowThreads + c;
        for (int i0 = 0; i0 < a; i0 += step) {
            uint4 v[kCommitRows];
#pragma unroll
            for (int i = 0; i < kCommitRows; ++i)
                if (i < step && i0 + i < a && s_src[i0 + i] >= 0) v[i] = pool[s_src[i0 + i] * kRowThreads];
#pragma unroll
            for (int i = 0; i < kCommitRows; ++i)
                if (i < step && i0 + i < a && s_src[i0 + i] >= 0) pool[s_dst[i0 + i] * kRowThreads] = v[i];
        }
    }
    // the kept length: the prefix, the root and the a accepted nodes (every
    // thread has read L: the barriers above)
    if (tid == 0) p.ctx_lens[b] = max(0, base + 1 + a);
}

}  // namespace

cs_status launch_kv_commit_tree(const cs_attn_dims& d, void* k_pages, void* v_pages, const int32_t* page_table,
                                int32_t* ctx_lens, const int32_t* path, const int32_t* n_accepted, int n_nodes,
                                cudaStream_t stream) {
    TreeCommitParams p{};
    p.k_pages = static_cast<uint4*>(k_pages);
    p.v_pages = static_cast<uint4*>(v_pages);
    p.page_table = page_table;
    p.ctx_lens = ctx_lens;
    p.path = path;
    p.n_accepted = n_accepted;
    p.n = n_nodes;
    p.Hkv = d.n_kv_heads;
    p.ps = d.page_size;
    p.max_pages = d.max_pages_per_seq;
    p.P = d.num_pages;
    // a thread for each column, and one for each node when there is one head
    const int heads = d.n_kv_heads < 32 ? d.n_kv_heads : 32;
    const int threads = heads > 1 ? heads * 2 * kRowThreads : CS_MAX_TREE_NODES;
    static_assert(32 * 2 * kRowThreads == kCommitMaxThreads && 2 * 2 * kRowThreads >= CS_MAX_TREE_NODES, "");
    const cudaError_t e =
        launch_dependent(kv_commit_tree_kernel, dim3(d.batch), dim3(threads), 0, stream, p);
    if (e != cudaSuccess) return cuda_fail(e, "kv_commit_tree_kernel launch");
    return CS_OK;
}

cs_status launch_kv_append(const cs_attn_dims& d, const void* new_k, const void* new_v, void* k_pages,
                           void* v_pages, const int32_t* page_table, const int32_t* ctx_lens, int n_new,
                           cudaStream_t stream) {
    AppendParams p{};
    p.new_k = static_cast<const uint4*>(new_k);
    p.new_v = static_cast<const uint4*>(new_v);
    p.k_pages = static_cast<uint4*>(k_pages);
    p.v_pages = static_cast<uint4*>(v_pages);
    p.page_table = page_table;
    p.ctx_lens = ctx_lens;
    p.rows = (long long)d.batch * n_new * d.n_kv_heads;
    p.n_new = n_new;
    p.Hkv = d.n_kv_heads;
    p.ps = d.page_size;
    p.max_pages = d.max_pages_per_seq;
    p.P = d.num_pages;
    const long long threads = p.rows * kRowThreads;
    const long long blocks = (threads + kAppendThreads - 1) / kAppendThreads;
    if (blocks > 0x7fffffffLL) return fail(CS_ERR_UNSUPPORTED, "too many rows to append in one call");
    const cudaError_t e =
        launch_dependent(kv_append_kernel, dim3((unsigned)blocks), dim3(kAppendThreads), 0, stream, p);
    if (e != cudaSuccess) return cuda_fail(e, "kv_append_kernel launch");
    return CS_OK;
}

cs_status launch_kv_commit(int32_t* ctx_lens, const int32_t* n_accepted, int batch, int n_draft,
                           cudaStream_t stream) {
    const cudaError_t e = launch_dependent(kv_commit_kernel, dim3((batch + 255) / 256), dim3(256), 0, stream,
                                           ctx_lens, n_accepted, batch, n_draft);
    if (e != cudaSuccess) return cuda_fail(e, "kv_commit_kernel launch");
    return CS_OK;
}

}  // namespace cs
