// Shared device/host helpers of libowlverify: work partition of the split-KV pass,
// status reporting, small PTX wrappers.  sm_100a only.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace owl {

constexpr int kHeadDim = 128;
constexpr int kMaxNodes = 64;     // drafted nodes per sequence (the paper's trees have 60)
constexpr int kMaxBatch = 1024;   // sequences per call (schedule prefix sums live in shared memory)
constexpr int kMaxRows = 256;     // packed rows (query heads of a KV group x nodes) per (sequence, KV head)

// Device-detected status codes: same values as owl_status in owlverify.h.
constexpr int kErrBadTree = -4;
constexpr int kErrBadPage = -5;
constexpr int kErrTimeout = -6;

struct SchedHeader;

// In the place of a partial's LSE: the pass met a malformed tree or a page out of range, the row stays unwritten.  A NaN that
// no arithmetic produces.  (It travels with the partial, so nothing is left over from one call for the next, and no call
// number has to tell the calls apart - a call replayed from a graph would carry the same one every time.)
constexpr uint32_t kBadPartial = 0x7fb0bad0u;

// Problem description handed to every kernel of the attention path.
struct AttnParams {
    const __nv_bfloat16* q;
    const __nv_bfloat16* k_cache;
    const __nv_bfloat16* v_cache;
    const int32_t* block_table;
    const int32_t* ctx_lens;
    const int32_t* node_offsets;  // may be null: uniform nodes_uniform per sequence
    const int32_t* tree_parent;
    __nv_bfloat16* out;
    float* lse;                   // may be null
    float* part_o;                // [slots, D / 4, kMaxRows, 4] fp32, normalised partial outputs
    float* part_lse;              // [slots, kMaxRows] fp32, natural-log partial LSE (-inf if empty; kBadPartial)
    int32_t* status;              // device status word (0 = ok, first error wins)
    long long* sched_seq_begin;   // [B + 1] first flat tile of every sequence (written by CTA 0 of the pass)
    SchedHeader* sched_header;
    int32_t batch, total_nodes, nodes_uniform, max_nodes;
    int32_t num_q_heads, num_kv_heads, group;  // group = Hq / Hkv
    uint32_t group_magic;         // 65536 / group + 1 (row_node)
    int32_t page_size, page_shift, max_pages_per_seq, num_pages;
    int32_t small;                // the schedule is derived by single warps in 32-bit arithmetic (small_schedule)
    int32_t num_ctas;             // CTAs of the split-KV pass (the flat tile range is cut into this many pieces)
    int32_t combine_group;        // partials per round of the merge kernel, 4..32
    int32_t combine_lg_parts;     // log2 of the CTAs that share a block's channels
    int32_t combine_row_ctas;     // the merge kernel's CTAs that take rows (persistent)
    int32_t f16;                  // q / caches / out are fp16 instead of bf16 (same size; typed as bf16 pointers here)
    float sm_scale;
};

// Node of a unit's packed row, row < kMaxRows.  (group * magic = 65536 + e with 1 <= e <= group, so the product is
// row / group + row * e / (65536 group), too high by less than 1 / group while row * group < 65536.)
__device__ __forceinline__ unsigned row_node(const AttnParams& p, unsigned row) { return (row * p.group_magic) >> 16; }

// 2^x by the special-function unit (ex2.approx, denormals flushed); ex2(-inf) = 0.
__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void report(int32_t* status, int code) { atomicCAS(status, 0, code); }

// ---------------------------------------------------------------------------------------------
// Partition of the split-KV pass.
//
// A unit is (sequence b, KV head h) with all its G * n_b packed rows; it owns
// tiles_b = ceil((L_b + n_b) / TileKeys) key tiles.  Units are laid out sequence-major, then head, on one line, which
// is cut into num_ctas contiguous pieces, one per CTA.  A piece may start and end inside a unit; only its first and its
// last unit can be cut, so a CTA stores at most two partials (o, lse): slot 2c for the unit its piece starts in, 2c + 1
// for a later one.
//   flat:    pieces of (nearly) equal length.  On the line a unit is `pen` = kBoundaryPenaltyTiles longer than its tiles,
//            the gap lying in front of them: what it costs a CTA to go from one unit to the next (pipeline drain,
//            epilogue, new Q: 6.8 us at 1.23 us per tile for units of up to 128 rows, 12.3 at 2.0 for 256).  With pieces
//            of equally many tiles the CTAs that held many short units ended last by far: 48 sequences of 200 to 6000
//            tokens 83 to 130 us, 4 x 128K 441 to 493 us.
//   aligned: only when every unit has the same number of tiles (`unit_tiles`) and there are at least as
//            many CTAs as units: unit u is cut into base + (u < urem) nearly equal pieces, so no piece
//            crosses a unit boundary (and there are no gaps).  Chosen when its largest piece is smaller than the flat one.
// ---------------------------------------------------------------------------------------------
constexpr int kBoundaryPenaltyTiles = 5;
// T: places on the line.  int where the host has made sure that the line is short (small_schedule).  Every CTA derives its
// piece once, on its critical path, where the code is not in the instruction caches and one instruction waits for the one
// before: instructions are time there.

// x / d for 0 <= x < 2^24, 0 < d and a quotient below 2^21: both are exact in fp32, the quotient of __fdividef (2 ulp) is off by
// less than one, and the remainder says which way.  Half the instructions of an integer division.
__host__ __device__ __forceinline__ int div_small(int x, int d) {
#ifdef __CUDA_ARCH__
    int q = (int)__fdividef((float)x, (float)d);
#else
    int q = x / d;
#endif
    const int r = x - q * d;
    if (r < 0) --q;
    if (r >= d) ++q;
    return q;
}

template <typename T>
struct Partition {
    static constexpr bool kShort = sizeof(T) == 4;
    T total, q;                   // length of the line, of a piece
    int rem, ctas;
    int unit_tiles, base, urem;   // aligned mode iff unit_tiles > 0
    int pen;                      // gap in front of a unit's tiles
    static __host__ __device__ __forceinline__ T div(T x, T d) {
        if constexpr (kShort) return div_small(x, d);
        else if (x >= 0 && x <= 0x7fffffffll && d <= 0x7fffffffll) return (T)((unsigned)x / (unsigned)d);
        else return x / d;
    }
    __host__ __device__ __forceinline__ void init(T tiles, int ctas_, int units, int uniform_tiles) {
        ctas = ctas_;
        pen = kBoundaryPenaltyTiles;
        total = tiles + (T)pen * units;
        q = div(total, ctas);
        rem = (int)(total - q * ctas);
        unit_tiles = 0; base = 0; urem = 0;
        if (uniform_tiles > 0 && units > 1 && units <= ctas) {
            const int b = (int)div(ctas, units);
            if (div((T)uniform_tiles + b - 1, b) < q + (rem ? 1 : 0)) {
                unit_tiles = uniform_tiles; base = b; urem = ctas - b * units;
                total = tiles; pen = 0;
            }
        }
    }
    // piece c, [t_begin, t_end)
    __host__ __device__ __forceinline__ void range(int c, T& t_begin, T& t_end) const {
        if (unit_tiles == 0) {
            t_begin = (T)c * q + min(c, rem);
            t_end = t_begin + q + (c < rem ? 1 : 0);
            return;
        }
        // the first urem units have one piece more
        const int big = urem * (base + 1), cu = c < big ? base + 1 : base;
        const int x = c < big ? c : c - big, u = (int)div(x, cu), k = x - u * cu;
        const int qq = (int)div(unit_tiles, cu), rr = unit_tiles - qq * cu;
        t_begin = (T)(c < big ? u : urem + u) * unit_tiles + (T)k * qq + min(k, rr);
        t_end = t_begin + qq + (k < rr ? 1 : 0);
    }
    __host__ __device__ __forceinline__ int owner(T t) const {      // of a place on the line
        T x = t, head = (T)rem * (q + 1), d = q;             // pieces, the first rem of them of d + 1 places
        int first = 0, longer = rem;
        if (unit_tiles > 0) {
            const int u = (int)div(t, unit_tiles), cu = base + (u < urem ? 1 : 0);
            x = t - (T)u * unit_tiles;
            first = u * base + min(u, urem);
            d = div(unit_tiles, cu);
            longer = unit_tiles - (int)d * cu;
            head = (T)longer * (d + 1);
        }
        return first + (x < head ? (int)div(x, d + 1) : longer + (int)div(x - head, d));
    }
};

// What the split-KV pass leaves for the combine kernel: totals and the choice of partition.
struct SchedHeader {
    long long total_tiles;   // of all units, without gaps
    int uniform_tiles;   // tiles per unit if every schedulable sequence has the same count, else 0
    int units;
};

__device__ __forceinline__ int seq_nodes(const AttnParams& p, int b) {
    return p.node_offsets ? p.node_offsets[b + 1] - p.node_offsets[b] : p.nodes_uniform;
}
__device__ __forceinline__ int seq_node_base(const AttnParams& p, int b) {
    return p.node_offsets ? p.node_offsets[b] : b * p.nodes_uniform;
}

// Loads of a call's inputs before the kernel's own dependency wait (the merge's schedule, the walk's tree, the cell's states).
// They may stand there because the kernel before it in the call lets its dependents start only after its own wait, when
// everything before the call has completed, and because that kernel writes none of them.  They take what L2 holds: an input
// that an earlier kernel wrote in place (lengths, z) may lie in the L1 of this SM as it was.
template <typename T>
__device__ __forceinline__ T ld_early(const T* p) { return __ldcg(p); }

// A sequence is schedulable when its node count and lengths are inside the interface's limits.
__device__ __forceinline__ bool seq_tree_shape_ok(const AttnParams& p, int base, int n) {
    return n >= 1 && n <= p.max_nodes && base >= 0 && base + n <= p.total_nodes;
}
__device__ __forceinline__ bool seq_shape_ok(const AttnParams& p, int b, int n, int L) {
    if (!seq_tree_shape_ok(p, seq_node_base(p, b), n) || L < 0) return false;
    long long keys = (long long)L + n;
    return keys <= (long long)p.max_pages_per_seq * p.page_size;
}

// Schedule of a batch of at most 32 sequences, derived by one warp on its own: lane b holds sequence b, prefix sums
// by shuffle, no shared memory.  The split-KV pass (its producer warp) and the merge that follows it (every warp) call the
// same function on the same inputs, so the merge needs nothing from the pass but its partials.
// The line is so short that everything fits 32 bits, a sequence's keys (2^24 tiles) included.
constexpr int kSchedTileKeys = 128;      // key tile of the split-KV pass
inline bool small_schedule(int batch, int num_kv_heads, int max_pages_per_seq, int page_size) {
    const long long tiles = ((long long)max_pages_per_seq * page_size + kSchedTileKeys - 1) / kSchedTileKeys;
    return batch <= 32 && (tiles + kBoundaryPenaltyTiles) * batch * num_kv_heads < (1ll << 24);
}
struct WarpSchedule {
    int n, L, node_base, tiles;          // this lane's sequence (tiles = 0 if it is not schedulable)
    unsigned ok;                         // the schedulable sequences
    int begin, end;                      // this lane's sequence on the line
    Partition<int> part;
};
__device__ __forceinline__ WarpSchedule warp_schedule(const AttnParams& p) {
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    WarpSchedule ws;
    ws.n = 0; ws.L = 0; ws.node_base = 0;
    bool ok = false;
    if (lane < p.batch) {
        ws.L = ld_early(p.ctx_lens + lane);
        ws.node_base = p.node_offsets ? ld_early(p.node_offsets + lane) : lane * p.nodes_uniform;
        ws.n = p.node_offsets ? ld_early(p.node_offsets + lane + 1) - ws.node_base : p.nodes_uniform;
        ok = seq_tree_shape_ok(p, ws.node_base, ws.n) && ws.L >= 0 &&
             (unsigned)ws.L + (unsigned)ws.n <= (unsigned)p.max_pages_per_seq * (unsigned)p.page_size;
    }
    ws.tiles = ok ? (ws.L + ws.n + kSchedTileKeys - 1) / kSchedTileKeys : 0;
    ws.ok = __ballot_sync(kAll, ok);
    const int first_tiles = __shfl_sync(kAll, ws.tiles, ws.ok ? __ffs(ws.ok) - 1 : 0);
    const bool uniform = __all_sync(kAll, !ok || ws.tiles == first_tiles);
    // tiles of one KV head's units; as many rounds as the batch needs
    int inc = ws.tiles;
    for (int o = 1; o < p.batch; o <<= 1) {
        const int v = __shfl_up_sync(kAll, inc, o);
        if (lane >= o) inc += v;
    }
    ws.part.init(__shfl_sync(kAll, inc, p.batch - 1) * p.num_kv_heads, p.num_ctas, __popc(ws.ok) * p.num_kv_heads, uniform ? first_tiles : 0);
    ws.end = (inc + ws.part.pen * __popc(ws.ok & (kAll >> (31 - lane)))) * p.num_kv_heads;
    ws.begin = ws.end - (ok ? (ws.tiles + ws.part.pen) * p.num_kv_heads : 0);
    return ws;
}

}  // namespace owl
