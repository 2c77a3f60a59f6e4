// The steps of the decoding loop on either side of the verify pass (Algorithm 1):
//   prepare_spec_kernel   Prepare(d): one [SPEC] leaf after every tree path, parents (= attention mask),
//                         depth-based position ids (Section 3.2.2 "Decode Stage")
//   kv_commit_kernel      "l <- l; d", "N <- N + |d|": the accepted nodes' K/V move from logical position
//                         L + path[k] to L + k in the paged cache, the committed length grows by accept_len
// Both are tiny and latency-bound: one CTA per sequence (and per KV head and cache for the move).
#pragma once

#include "owl_common.cuh"

namespace owl {

struct PrepareParams {
    const int32_t* node_offsets;   // may be null: nodes_uniform drafted nodes per sequence
    const int32_t* tree_parent;
    const int32_t* draft_tokens;
    const int32_t* ctx_lens;
    const int32_t* route;          // may be null (every sequence gets [SPEC] leaves); route[b] == 0: chain kept as drafted
    int32_t* out_offsets;          // [B + 1]: running sum of the output node counts (n or 2 n per sequence)
    int32_t* out_parent;           // [2 N]
    int32_t* out_draft;            // [2 N], -1 for a [SPEC] leaf
    int32_t* out_input_ids;        // [2 N], spec_token for a [SPEC] leaf
    int32_t* out_position;         // [2 N], ctx_len + depth
    int32_t* status;
    int32_t batch, total_nodes, nodes_uniform, max_nodes, spec_token;
};

constexpr int kPrepareThreads = 64;
static_assert(kPrepareThreads >= kMaxNodes, "one thread per drafted node");

// One CTA per sequence, one thread per drafted node j: node j keeps its place, its [SPEC] leaf is node n + j.
// With a route array, a sequence routed to non-tree verification (route 0) keeps its chain without any [SPEC]
// (Section 3.2.3); the sequences' outputs are packed one after the other, so every CTA first sums the output
// node counts of the sequences before its own.
__global__ void __launch_bounds__(kPrepareThreads) prepare_spec_kernel(const PrepareParams p) {
    // may be launched as a programmatic dependent: nothing is read before the kernel before it in the stream has
    // completed (a no-op in an ordinary launch); the kernel after this one may queue up and waits likewise
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // Two rounds of loads, everything that does not need the offsets in the first.
    const int b = blockIdx.x, j = threadIdx.x;
    const int base = p.node_offsets ? p.node_offsets[b] : b * p.nodes_uniform;
    const int n = p.node_offsets ? p.node_offsets[b + 1] - base : p.nodes_uniform;
    const bool with_spec = !p.route || p.route[b] != 0;
    const int L = p.ctx_lens[b];
    __shared__ int s_parent[kMaxNodes];
    __shared__ int s_before[2];
    int before = 0;                  // output nodes of sequences 0 .. b-1
    if (p.route) {
        for (int c = j; c < b; c += kPrepareThreads) {
            const int nc = p.node_offsets ? p.node_offsets[c + 1] - p.node_offsets[c] : p.nodes_uniform;
            before += p.route[c] != 0 ? 2 * nc : nc;
        }
        before = __reduce_add_sync(0xffffffffu, before);
        if ((j & 31) == 0) s_before[j >> 5] = before;
    }
    const bool mine = n >= 1 && n <= p.max_nodes && j < n && base >= 0 && base + n <= p.total_nodes;
    int parent = -1, tok = 0;
    if (mine) {
        parent = p.tree_parent[base + j];
        tok = p.draft_tokens[base + j];
    }
    s_parent[j] = parent;
    bool bad = mine && (j == 0 ? parent != -1 : parent < 0 || parent >= j);
    bad = __syncthreads_or(bad);
    const int ob = p.route ? s_before[0] + s_before[1] : 2 * base, count = with_spec ? 2 * n : n;
    if (j == 0) {
        if (b == 0) p.out_offsets[0] = 0;
        p.out_offsets[b + 1] = ob + count;
    }
    // the outputs hold 2 * total_nodes entries: whatever the offsets say, nothing is written outside them
    bad = bad || n < 1 || n > p.max_nodes || count > kMaxNodes || base < 0 || base + n > p.total_nodes || ob < 0 ||
          (long long)ob + count > 2ll * p.total_nodes;
    if (bad) { if (j == 0) report(p.status, kErrBadTree); return; }     // nothing of this sequence is written
    if (j < n) {
        int depth = 0;
        for (int c = parent; c >= 0; c = s_parent[c]) ++depth;          // parents come first: it ends
        const int o = ob + j;
        p.out_parent[o] = parent;
        p.out_draft[o] = tok;
        p.out_input_ids[o] = tok;
        p.out_position[o] = L + depth;
        if (with_spec) {
            p.out_parent[o + n] = j;
            p.out_draft[o + n] = -1;
            p.out_input_ids[o + n] = p.spec_token;
            p.out_position[o + n] = L + depth + 1;
        }
    }
}

struct CommitParams {
    __nv_bfloat16* k_cache;
    __nv_bfloat16* v_cache;
    const int32_t* block_table;
    int32_t* ctx_lens;             // in / out
    const int32_t* node_offsets;   // may be null
    const int32_t* accept_len;
    const int32_t* accept_path;
    int32_t* status;
    int32_t batch, total_nodes, nodes_uniform, max_nodes, num_kv_heads;
    int32_t page_size, page_shift, max_pages_per_seq, num_pages, path_stride;
};

constexpr int kCommitThreads = 256;      // half of them move K, half V
constexpr int kCommitMaxCluster = 8;     // CTAs of a sequence
constexpr int kCommitPages = 6;          // 64 drafted positions on pages of at least 16 touch five at most

// What every CTA of sequence b decides alike, from the inputs alone: 0 = commit, else the error code.
// The accepted path must be a root path in node order (path[0] = 0, strictly increasing, below n) and every page
// the drafted positions L .. L + n - 1 touch must exist: s_pages[i], the i-th of them, and s_path are the sequence's
// afterwards.  Called by all threads of a CTA (two barriers).  The path is read along with the lengths, before it is known how
// much of it counts.
__device__ __forceinline__ int commit_verdict(const CommitParams& p, int b, int& L, int& n, int& a, int* s_path /*[kMaxNodes]*/,
                                              int* s_pages /*[kCommitPages]*/) {
    const int t = threadIdx.x;
    const int base = p.node_offsets ? p.node_offsets[b] : b * p.nodes_uniform;
    n = p.node_offsets ? p.node_offsets[b + 1] - base : p.nodes_uniform;
    L = p.ctx_lens[b];
    a = p.accept_len[b];
    int v = 0, prev = -1;
    if (t < kMaxNodes && t < p.path_stride) {
        v = p.accept_path[(long long)b * p.path_stride + t];
        if (t > 0) prev = p.accept_path[(long long)b * p.path_stride + t - 1];
    }
    const bool shape_ok = n >= 1 && n <= p.max_nodes && n <= kMaxNodes && a >= 1 && a <= n && a <= p.path_stride && L >= 0 &&
                          (long long)L + n <= (long long)p.max_pages_per_seq * p.page_size;
    if (!shape_ok) return kErrBadTree;
    const bool bad_path = t < a && ((t == 0 && v != 0) || v <= prev || v >= n);
    if (t < a) s_path[t] = v;
    const int first_page = L >> p.page_shift, last_page = (L + n - 1) >> p.page_shift;
    bool bad_page = false;
    if (t <= last_page - first_page) {
        const int pg = p.block_table[(long long)b * p.max_pages_per_seq + first_page + t];
        bad_page = (unsigned)pg >= (unsigned)p.num_pages;
        s_pages[t] = pg;
    }
    const int verdict = __syncthreads_or(bad_path ? 1 : 0) ? kErrBadTree : 0;
    return __syncthreads_or(bad_page ? 1 : 0) && !verdict ? kErrBadPage : verdict;
}

// grid (C, B) in clusters of (C, 1), C = min(Hkv, 8): a sequence's heads are dealt out to its cluster's CTAs.  Every source
// row is read into shared memory before any destination is written, because a position can be the source of one move and
// the destination of a later one.  The committed length grows by accept_len once all CTAs of the sequence have read the old
// one: the cluster's barrier says so, and nothing is kept from one call for the next (a counter per sequence in the
// context did the same for one stream at a time; a second kernel for the lengths is one more launch in the chain).
__global__ void __launch_bounds__(kCommitThreads) kv_commit_kernel(const CommitParams p) {
    // may be launched as a programmatic dependent: nothing is read before the kernel before it in the stream has
    // completed (a no-op in an ordinary launch); the kernel after this one may queue up and waits likewise
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ uint4 s_rows[2][kMaxNodes * 16];    // up to 64 rows of 128 bf16 each of K and V
    __shared__ int s_path[kMaxNodes];
    __shared__ int s_pages[kCommitPages];
    const int b = blockIdx.y;
    int L, n, a;
    const int verdict = commit_verdict(p, b, L, n, a, s_path, s_pages);
    if (verdict != 0) {                            // in every CTA of the cluster
        if (threadIdx.x == 0 && blockIdx.x == 0) report(p.status, verdict);
        return;
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");      // this CTA has read the length
    const int kv = threadIdx.x / (kCommitThreads / 2), first = (threadIdx.x % (kCommitThreads / 2)) >> 4, piece = threadIdx.x & 15;
    constexpr int kStep = kCommitThreads / 32;     // rows per turn of a half
    __nv_bfloat16* cache = kv ? p.v_cache : p.k_cache;
    const int first_page = L >> p.page_shift;
    for (int h = blockIdx.x; h < p.num_kv_heads; h += gridDim.x) {
        auto row_ptr = [&](int pos) {
            const long long page = s_pages[(pos >> p.page_shift) - first_page];
            return reinterpret_cast<uint4*>(cache + ((page * p.num_kv_heads + h) * p.page_size + (pos & (p.page_size - 1))) * kHeadDim);
        };
        for (int k = first; k < a; k += kStep)
            if (s_path[k] != k) s_rows[kv][k * 16 + piece] = row_ptr(L + s_path[k])[piece];
        __syncthreads();
        for (int k = first; k < a; k += kStep)         // (a thread takes back what it put there itself)
            if (s_path[k] != k) row_ptr(L + k)[piece] = s_rows[kv][k * 16 + piece];
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (blockIdx.x == 0 && threadIdx.x == 0) p.ctx_lens[b] = L + a;
}

}  // namespace owl
