// Greedy tree acceptance: row arg-max over the vocabulary, then the acceptance walk.
//
// The scan reads fp32 logits with 16-byte loads, one warp per (row, vocabulary chunk of 2048 to 8192 floats) item.  Every
// (value, index) candidate is folded into one 64-bit key, high word = the float mapped to an unsigned
// integer that sorts like the float (NaN mapped to -inf, -0 to +0), low word = ~index, so that an unsigned
// max picks the larger value and, among equal values, the lower index.  Per-lane and warp (shuffle) maxima
// give one key per item, stored to part_keys[row][chunk] (no atomics, nothing to initialise).
//
// The walk reduces the chunk keys to arg-max tokens, evaluates for every node whether all edges on its
// root path match (draft token == parent's arg-max), picks the deepest matching node (lowest index among
// equals) and writes accept_len / accept_path / bonus_token.  It follows the scan as a kernel of its own (one CTA per
// sequence), in a verify step as extra CTAs of the merge kernel.  (The scan used to count its items per sequence, and
// the CTA that completed one walked its tree: the fence and the atomic after every item cost 1.35 us each with the
// warp's loads drained, 7 of the 68 us of a 756-row scan.)
//
// Inside a verify step with a small scan both halves run as guests of the attention kernels: the scan in warps
// the attention pass does not use (argmax_scan_chunk_warp), the walk in extra CTAs of the merge kernel, after
// the pass has completed.
#pragma once

#include "owl_common.cuh"

namespace owl {

constexpr int kArgmaxThreads = 256;
static_assert(kArgmaxThreads >= kMaxNodes, "the walk needs one thread per node");
constexpr int kArgmaxChunk = 8192;     // floats per item when there are items enough for every warp
constexpr int kArgmaxMinChunk = 2048;  // two rounds of eight 16-byte loads per lane
// Floats per (row, chunk) item of a scan by `warps` warps: halved as long as every warp still gets one item at most.  A
// small scan is bound by the loads a warp can keep in flight, so it needs all the warps (60 rows x 128256: 960 items of
// 8192 kept 960 of 2368 warps busy).
__host__ inline int argmax_chunk(long long rows, int vocab, long long warps) {
    int chunk = kArgmaxChunk;
    while (chunk > kArgmaxMinChunk && rows * ((vocab + chunk / 2 - 1) / (chunk / 2)) <= warps) chunk /= 2;
    return chunk;
}

// 16-byte load of data that is read once: no L1 allocation, first in line for eviction from L2
// (`policy` from createpolicy.fractional.L2::evict_first).
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ float4 ld_stream_f4(const float4* ptr, uint64_t policy) {
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(ptr), "l"(policy));
    return v;
}

struct AcceptParams {
    const float* logits;
    const int32_t* draft_tokens;
    const int32_t* node_offsets;
    const int32_t* tree_parent;
    int32_t* accept_len;
    int32_t* accept_path;
    int32_t* bonus_token;
    int32_t* node_argmax;
    int32_t* spec_node;              // optional [B]: the [SPEC] leaf (negative draft token) under the last accepted node
    unsigned long long* part_keys;   // [total_nodes, chunks]
    int32_t early;                   // the kernel before this one in the stream is the attention pass of the same step
    int32_t* status;
    int32_t batch, total_nodes, nodes_uniform, max_nodes, vocab, path_stride;
    int32_t chunk, chunks;           // floats per item, items per row
};

// The LM-head product's row keys only ever grow (atomicMax) and must start from 0, below every real key.  Two sets of
// `stride` keys alternate between calls: a call's product raises one, its walk reads that one and clears the other as a
// whole, so that no memset stands in front of a product.  Which set is a call's own is counted on the device - a call
// replayed from a graph has its host side behind it: the product reads call[0] and leaves what it read in call[1], the
// walk goes by call[1] and moves call[0] on.  (Two words, because a walk's CTAs read the number while one of them moves it.)
struct KeySets {
    unsigned long long* keys;        // [2, stride]
    uint32_t* call;
    int32_t stride;
};

__device__ __forceinline__ unsigned long long argmax_key(float x, uint32_t idx) {
    if (x != x) x = -INFINITY;   // NaN never wins
    x += 0.0f;                   // -0.0 -> +0.0
    uint32_t u = __float_as_uint(x);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((unsigned long long)u << 32) | (uint32_t)(~idx);
}

// The kernel before this one in the stream has completed and its writes are visible; the next one may queue up.
__device__ __forceinline__ void wait_and_let_dependents_start() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// One sequence's walk; called by the first kArgmaxThreads threads of a CTA.  A node's chunk keys are read by several
// neighbouring threads, all in one memory round trip; the rest is the first warp's, two nodes per lane.
// `keys()` waits for the kernel that leaves the arg-max keys and returns them.  The tree and the tokens are read before
// (ld_early).  With the ancestors as bits by then, what is left when the keys are there is one round of loads, one CTA barrier
// and a handful of votes.
template <typename Keys>
__device__ __forceinline__ void accept_walk_seq(const AcceptParams& p, const int b, Keys keys) {
    constexpr unsigned kAll = 0xffffffffu;
    static_assert(kMaxNodes == 64, "two nodes per lane of a warp");
    static_assert(kArgmaxThreads >= 4 * kMaxNodes, "at least four threads per node");
    __shared__ int s_parent[kMaxNodes], s_am[kMaxNodes];
    const int i = threadIdx.x, lane = i & 31;
    const int base = p.node_offsets ? ld_early(p.node_offsets + b) : b * p.nodes_uniform;
    const int n = p.node_offsets ? ld_early(p.node_offsets + b + 1) - base : p.nodes_uniform;
    const bool shape_ok = n >= 1 && n <= p.max_nodes && n <= p.path_stride && base >= 0 && base + n <= p.total_nodes;
    int parent[2] = {-1, -1}, tok[2] = {-1, -1};
    unsigned long long anc[2] = {0ull, 0ull};          // the node and its ancestors
    bool bad = false;
    if (i < 32 && shape_ok) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int node = lane + 32 * h;
            if (node >= n) continue;
            parent[h] = ld_early(p.tree_parent + base + node);
            tok[h] = ld_early(p.draft_tokens + base + node);
            bad = bad || (node == 0 ? parent[h] != -1 : parent[h] < 0 || parent[h] >= node);
            s_parent[node] = parent[h];
        }
        bad = __any_sync(kAll, bad);
        __syncwarp();                                  // a vote orders no memory: the lanes' parents are there, and checked
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (!bad && lane + 32 * h < n)
                for (int c = lane + 32 * h; c >= 0; c = s_parent[c]) anc[h] |= 1ull << c;      // parents come first: it ends
    }
    const unsigned long long* part_keys = keys();
    if (!shape_ok) { if (i == 0) report(p.status, kErrBadTree); return; }
    {
        const int lg = n > 32 ? 2 : n > 16 ? 3 : n > 8 ? 4 : 5;       // 4 to 32 threads per node
        const int node = i >> lg, sub = i & ((1 << lg) - 1);
        unsigned long long k = 0;
        if (node < n) {
            const unsigned long long* pk = part_keys + (long long)(base + node) * p.chunks;
            for (int c0 = sub; c0 < p.chunks; c0 += 8 << lg) {
                unsigned long long v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = c0 + (j << lg) < p.chunks ? __ldcg(pk + c0 + (j << lg)) : 0ull;
#pragma unroll
                for (int j = 0; j < 8; ++j) k = v[j] > k ? v[j] : k;
            }
        }
        for (int o = (1 << lg) >> 1; o > 0; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(kAll, k, o);
            k = other > k ? other : k;
        }
        if (node < n && sub == 0) {
            const int am = (int)(~(uint32_t)(k & 0xffffffffull));
            s_am[node] = am;
            if (p.node_argmax) p.node_argmax[base + node] = am;
        }
    }
    asm volatile("bar.sync 0, %0;" ::"n"(kArgmaxThreads) : "memory");
    if (i >= 32) return;
    if (bad) { if (i == 0) report(p.status, kErrBadTree); return; }

    // a node is accepted if it and all its ancestors but the root are what the verifier chose at their parents
    unsigned long long match = 1ull;
#pragma unroll
    for (int h = 0; h < 2; ++h)
        match |= (unsigned long long)__ballot_sync(kAll, parent[h] >= 0 && tok[h] >= 0 && tok[h] == s_am[max(parent[h], 0)]) << (32 * h);
    unsigned best = 0;                                  // deepest, then lowest index
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (anc[h] && !(anc[h] & ~match)) best = max(best, (unsigned)__popcll(anc[h]) << 8 | (unsigned)(kMaxNodes - 1 - lane - 32 * h));
    best = __reduce_max_sync(kAll, best);
    const int win = kMaxNodes - 1 - (int)(best & 0xffu), len = (int)(best >> 8);
    const unsigned long long anc_win = __shfl_sync(kAll, win >= 32 ? anc[1] : anc[0], win & 31);
    int32_t* path = p.accept_path + (long long)b * p.path_stride;
#pragma unroll
    for (int h = 0; h < 2; ++h)                         // parents come first: a path is its nodes in ascending order
        if (anc_win >> (lane + 32 * h) & 1ull) path[__popcll(anc_win & ((1ull << (lane + 32 * h)) - 1ull))] = lane + 32 * h;
    for (int k = len + lane; k < p.path_stride; k += 32) path[k] = -1;
    // Section 3.2.2 "Decode Stage": the hidden state handed to the drafter is that of the [SPEC] which follows
    // the accepted path, i.e. the [SPEC] child of its last node (lowest index if several, -1 if none)
    const unsigned leaf0 = __ballot_sync(kAll, lane < n && parent[0] == win && tok[0] < 0);
    const unsigned leaf1 = __ballot_sync(kAll, lane + 32 < n && parent[1] == win && tok[1] < 0);
    if (lane == 0) {
        p.accept_len[b] = len;
        p.bonus_token[b] = s_am[win];
        if (p.spec_node) p.spec_node[b] = leaf0 ? __ffs(leaf0) - 1 : leaf1 ? __ffs(leaf1) + 31 : -1;
    }
}

// Scan of one (row, vocabulary chunk) item by a single warp: eight 16-byte loads per lane and round.  Per round a
// lane first takes the maximum of its 32 values by a tree of fmaxf (NaN drops out: fmaxf returns the other operand,
// and the final fmaxf with -inf turns an all-NaN round into -inf), and only if that beats its best so far - which
// becomes rare quickly - looks for the first value that attains it.  Strict '>' and first-match keep the lowest
// index among equal values, because a lane's indices grow along its walk; the maximum over (value, ~index) keys
// then does not depend on how the chunk's elements are dealt out to lanes.
// The next round's loads are issued before this round is reduced.
__device__ __forceinline__ void argmax_scan_chunk_warp(const AcceptParams& p, const int row, const int chunk) {
    const int lane = threadIdx.x & 31;
    const long long V = p.vocab;
    const long long c0 = (long long)chunk * p.chunk;
    const long long c1 = c0 + p.chunk < V ? c0 + p.chunk : V;
    const float* base = p.logits + row * V;
    // [c0, a0) scalar head up to 16-byte alignment, [a0, a1) float4 body, [a1, c1) scalar tail
    const uintptr_t addr = reinterpret_cast<uintptr_t>(base + c0);
    long long a0 = c0 + (long long)(((16 - (addr & 15)) & 15) >> 2);
    if (a0 > c1) a0 = c1;
    const long long a1 = a0 + ((c1 - a0) & ~3ll);

    float bv = -INFINITY;
    uint32_t bi = 0xffffffffu;   // "no candidate yet"
    const float4* body = reinterpret_cast<const float4*>(base + a0);
    const int nvec = (int)((a1 - a0) >> 2);
    const uint64_t policy = l2_evict_first_policy();     // the logits are read once
    const float4 none = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    auto load_round = [&](int v0, float4 (&x)[8]) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {            // eight independent 16-byte loads per lane in flight
            const int v = v0 + j * 32 + lane;
            x[j] = v < nvec ? ld_stream_f4(body + v, policy) : none;
        }
    };
    auto reduce_round = [&](int v0, const float4 (&x)[8]) {
        float m[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) m[j] = fmaxf(fmaxf(x[j].x, x[j].y), fmaxf(x[j].z, x[j].w));
        const float mx = fmaxf(fmaxf(fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])), fmaxf(fmaxf(m[4], m[5]), fmaxf(m[6], m[7]))), -INFINITY);
        if (v0 + lane < nvec && (bi == 0xffffffffu || mx > bv)) {
            // a new best (or the first candidate): the first of this round's values that attains it; slots past
            // the end hold -inf, which only an all -inf round matches, and then the round's first slot wins
            bv = mx;
#pragma unroll
            for (int j = 7; j >= 0; --j) {
                const uint32_t i0 = (uint32_t)(a0 + 4ll * (v0 + j * 32 + lane));
                if (fmaxf(x[j].w, -INFINITY) == mx) bi = i0 + 3;
                if (fmaxf(x[j].z, -INFINITY) == mx) bi = i0 + 2;
                if (fmaxf(x[j].y, -INFINITY) == mx) bi = i0 + 1;
                if (fmaxf(x[j].x, -INFINITY) == mx) bi = i0;
            }
        }
    };
    float4 xa[8], xb[8];
    if (nvec > 0) load_round(0, xa);
    for (int v0 = 0; v0 < nvec; v0 += 2 * 32 * 8) {
        if (v0 + 32 * 8 < nvec) load_round(v0 + 32 * 8, xb);
        reduce_round(v0, xa);
        if (v0 + 2 * 32 * 8 < nvec) load_round(v0 + 2 * 32 * 8, xa);
        if (v0 + 32 * 8 < nvec) reduce_round(v0 + 32 * 8, xb);
    }
    unsigned long long key = bi != 0xffffffffu ? argmax_key(bv, bi) : 0ull;
    if (lane < 8) {              // ragged ends: at most 3 + 3 elements per chunk
        const long long j = lane < 4 ? c0 + lane : a1 + (lane - 4);
        const long long lim = lane < 4 ? a0 : c1;
        if (j < lim) {
            const unsigned long long k2 = argmax_key(base[j], (uint32_t)j);
            key = k2 > key ? k2 : key;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, key, o);
        key = other > key ? other : key;
    }
    if (lane == 0) p.part_keys[(long long)row * p.chunks + chunk] = key;
}

// Persistent scan: the grid's warps take the (row, vocabulary chunk) items in turn (consecutive warps read
// consecutive chunks), each with up to two rounds of eight 16-byte loads per lane in flight, so that a warp streams
// without the per-item cost of a CTA's launch and barriers.
constexpr int kArgmaxWarps = kArgmaxThreads / 32;
constexpr int kScanAhead = 4096;        // floats
constexpr int kArgmaxCtasPerSm = 2;     // what fits at the kernel's register count; argmax_grid counts on it
__host__ inline long long argmax_warps(int sms) { return (long long)sms * kArgmaxCtasPerSm * kArgmaxWarps; }

__global__ void __launch_bounds__(kArgmaxThreads, kArgmaxCtasPerSm) argmax_partial_kernel(const AcceptParams p) {
    // may be launched as a programmatic dependent of the kernel before it in the stream: nothing is read
    // before that kernel has completed (a no-op in an ordinary launch).  After the attention pass of the same step the
    // scan need not wait: the pass lets its dependents start only once everything before it has completed, and the
    // scan reads nothing of the pass.  The CTAs then fill the SMs as their attention CTAs end (which is tens of
    // microseconds apart), and wait before they exit, so that the merge that follows finds the pass completed.
    if (!p.early && (threadIdx.x & 31) == 0) {
        // The warp's first rounds are asked for to L2 under the tail of whatever precedes this kernel (756 rows x 128256
        // 61.3 -> 59.3 us per call, 60 rows 9.1 -> 8.4).  It hands nothing to this kernel yet: L2 holds what was written last.
        const long long it = (long long)blockIdx.x * kArgmaxWarps + (threadIdx.x >> 5);
        if (it < (long long)p.total_nodes * p.chunks) {
            const long long row = it / p.chunks, c0 = (it - row * p.chunks) * p.chunk;
            const long long n = min((long long)min(p.chunk, kScanAhead), (long long)p.vocab - c0);
            const uintptr_t b = reinterpret_cast<uintptr_t>(p.logits + row * p.vocab + c0);
            const uintptr_t lo = (b + 15) & ~(uintptr_t)15, hi = (b + 4 * n) & ~(uintptr_t)15;
            if (hi > lo) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"((uint32_t)(hi - lo)) : "memory");
        }
    }
    if (!p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the next kernel may queue up (what it reads early: ld_early)
    const int warp = threadIdx.x >> 5;
    if (blockIdx.x == 0) {
        // Do the packed offsets describe this call's rows: start at 0, end at total_nodes, 1..max_nodes nodes per sequence?
        // (If not, the status word says so; the walks check what they touch.)
        if (p.node_offsets) {
            bool bad = false;
            for (int b = threadIdx.x; b < p.batch; b += kArgmaxThreads) {
                const int lo = p.node_offsets[b], n = p.node_offsets[b + 1] - lo;
                bad = bad || n < 1 || n > p.max_nodes || (b == 0 && lo != 0) || (b == p.batch - 1 && lo + n != p.total_nodes);
            }
            if (bad) report(p.status, kErrBadTree);
        }
    }
    const long long items = (long long)p.total_nodes * p.chunks;
    const long long stride = (long long)gridDim.x * kArgmaxWarps;
    for (long long it = (long long)blockIdx.x * kArgmaxWarps + warp; it < items; it += stride) {
        const int row = (int)(it / p.chunks), chunk = (int)(it - (long long)row * p.chunks);
        argmax_scan_chunk_warp(p, row, chunk);
    }
    if (p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// One sequence's acceptance walk per CTA over the keys the scan left.  Launched as a programmatic dependent of the scan.
__global__ void __launch_bounds__(kArgmaxThreads) accept_walk_kernel(const AcceptParams p) {
    accept_walk_seq(p, (int)blockIdx.x, [&] {
        wait_and_let_dependents_start();
        return (const unsigned long long*)p.part_keys;
    });
}
// The same over the keys of the LM-head product (a kernel of its own, so that the short acceptances do not carry the choice
// of the set).
__global__ void __launch_bounds__(kArgmaxThreads) accept_walk_sets_kernel(const AcceptParams p, const KeySets sets) {
    uint32_t call = 0;
    accept_walk_seq(p, (int)blockIdx.x, [&] {
        wait_and_let_dependents_start();
        call = __ldcg(sets.call + 1);
        return (const unsigned long long*)(sets.keys + (size_t)(call & 1u) * sets.stride);
    });
    unsigned long long* idle = sets.keys + (size_t)((call + 1u) & 1u) * sets.stride;
    for (int i = blockIdx.x * kArgmaxThreads + threadIdx.x; i < sets.stride; i += gridDim.x * kArgmaxThreads) idle[i] = 0ull;
    if (blockIdx.x == 0 && threadIdx.x == 0) sets.call[0] = call + 1u;
}

// Grid of the scan for `items` (row, chunk) items on a device with `sms` multiprocessors: as many warps as give
// every warp the same number of items (4096 items on 2368 resident warps would leave a quarter of the warps idle
// during the second half of the kernel; 2048 warps with two items each do not).
__host__ inline unsigned argmax_grid(long long items, int sms) {
    const long long max_warps = argmax_warps(sms);
    const long long rounds = (items + max_warps - 1) / max_warps;
    const long long warps = rounds > 0 ? (items + rounds - 1) / rounds : 1;
    const long long ctas = (warps + kArgmaxWarps - 1) / kArgmaxWarps;
    return (unsigned)(ctas < 1 ? 1 : ctas);
}

}  // namespace owl
