// Weight-streaming product C[M, N] = A[M, K] B[N, K]^T on the 5th-generation tensor cores (bf16 operands, fp32
// accumulators in tensor memory), for the two producers either side of the verify step:
//   LM head     A = hidden states of the drafted nodes [nodes, K], B = head weight [vocab, K]; the epilogue keeps of every
//               row of A only its arg-max over the vocabulary - the logits are never written;
//   drafter     A = h [rows, d_in], B = [W^f; W^i; W^o; W^c] ([4d, d_in]), Eq. 2; the epilogue stores fp32.
// M is small (up to 384 rows), N is huge: B is read from HBM exactly once, A comes again and again out of L2.
//
// The WEIGHTS are the instruction's M operand wherever a tile has more rows of B than there are rows of A (the other way
// round, kRowsOnLanes, is below): the accumulator is C^T, one row of B per lane of tensor memory, one row of A (rounded up
// to 16) per column.  What bounds the product is B's bytes and, run in a loop, the board's power.  With A as
// the M operand every instruction multiplied 128 rows however few exist: at 30 rows and 6 TB/s the tensor cores did the
// work of an 800 TFLOP/s product, three quarters of it on rows that nobody reads, and the power cap took the SM clock from
// 1965 to 1140 MHz, which slows the memory system as well.
//
// CTA pairs (cta_group::2) at every M: two CTAs on neighbouring SMs run one tcgen05.mma of M = 256 together.  CTA r stages
// half of the tile's rows of B (its own 128 accumulator lanes) and half of A's rows, so A is staged once per 256 rows of
// B and per SM half as often; each SM's tensor memory holds two accumulator buffers, so the epilogue of a tile hides under
// the next tile's products.  One thread issues for two SMs, and its time is the other limit: a wait, a commit and the loop
// around them cost it some 800 clocks a stage when written plainly (divisions by the ring's length, 64-bit descriptor
// arithmetic, one k-block a stage).  A stage holds two k-blocks (eight products per wait and commit), slot and phase run
// along as counters, and each thread looks at its next barrier before it needs it.
// Above 256 rows of A the accumulator is two groups of up to 192 columns in one buffer, a stage one k-block (the same
// eight products).
//
// Measured (128256 x 4096 weights, us in a loop at the power cap; before = A as the M operand): 16 rows 192 -> 161, 32 rows
// 195 -> 158, 64 rows 205 -> 163, 96 rows 195 -> 172, 128 rows 203 -> 183, 144 rows 281 -> 216, 192 rows 279 -> 233,
// 256 rows 286 -> 273.  One CTA per SM instead of pairs: 162 / 163 / 175 / 185 / 193 us at 16 / 32 / 64 / 96 / 128 rows.
//
// kRowsOnLanes: few weights and many rows (weights of a few MB cut over 74 pairs make tiles of 16 to 100 rows of B, and
// 256 rows of A as columns then keep the tensor cores busy for far longer than the bytes take).  The same stages, with the
// roles of the two operands swapped in the instruction: one row of A per lane, the tile's rows of B as columns; a thread
// of the epilogue owns a row of A for the whole kernel.  (rows_on_lanes has the rule and the figures.)
//
// Balance.  Every pair gets ceil(N / 16 / pairs) units of 16 rows of B, cut into as few tiles of at most 256 as
// possible, the tiles of one round equally high on every pair (heights differ by at most 16 between rounds).
// Ring.  At 6.5 TB/s over 148 SMs and 2.5-3 us of loaded memory latency a CTA needs 110-130 KB of B in flight, so a stage
// holds the tile's rows of B and A's rows and nothing else; a 128-row window on fewer rows runs on into whatever follows
// in shared memory, which feeds accumulator lanes that nobody reads.
// Roles (256 threads): warp 0 TMA producer (copies complete on the EVEN CTA's arrival barrier; no multicast), warp 1 of the
// even CTA issues, warps 4-7 epilogue (thread = lane of tensor memory = row of B).  Every wait is bounded; a wait that
// gives up raises both CTAs' abort flags.
#pragma once

#include <cuda.h>
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "accept.cuh"
#include "kv_tensor_map.cuh"
#include "owl_common.cuh"
#include "sm100_ptx.cuh"

namespace owl {
namespace gemm_path {

using namespace sm100;

enum Epilogue { kEpiArgmax = 0, kEpiStore = 1 };
constexpr uint32_t kNobody = 0xffffffffu;

constexpr int kBK = 64;                          // a k-block: one 128-byte swizzle row per operand row
constexpr int kThreads = 256;
constexpr int kWindowBytes = 128 * kBK * 2;      // what an instruction reads of one CTA's rows of B: 16 KB
constexpr int kMaxStages = 8;
constexpr int kAuxBytes = 4096;
constexpr int kSmemLimit = 232448;               // 227 KB
// A launch asks for at least this much, so that an SM never holds two of these CTAs (2 x (116 + 1) KB > 228 KB).  Each
// takes all of its SM's tensor memory, and a pair takes that of two SMs: two pairs of different streams on the same two
// SMs, each with one half allocated, would wait for each other for good.
constexpr int kSmemAlone = 118784;
constexpr int kMaxTile = 256;                    // rows of B per tile, both CTAs
constexpr int kMaxRows = 384;                    // rows of A
constexpr int kGroupRows = 256;                  // rows of A in one column group; above, two groups

struct GemmParams {
    int M, N, K;
    int group_rows;                 // rows of A per column group, a multiple of 16: the instruction's N
    int stages;
    int block_bytes;                // a k-block of a stage: this CTA's rows of B, then its rows of A, 128 bytes each
    int rounds;                     // tiles per pair; all tiles of a round are equally high
    int tall_rounds;                // rounds [0, tall_rounds) are h_lo + 16 rows of B high, the others h_lo
    int h_lo;                       // multiple of 16, <= 256
    int32_t* status;
    KeySets sets;                   // kEpiArgmax: keys (value, ~column) of the rows, raised by atomicMax
    float* c;                       // kEpiStore: fp32 [M, ldc]
    long long ldc;
};

struct Aux {
    uint64_t full[kMaxStages], empty[kMaxStages];   // `full` is used in the even CTA only
    uint64_t acc_full[2], acc_empty[2];             // `acc_empty` is used in the even CTA only (256 arrivals)
    unsigned long long best[kMaxRows];              // kEpiArgmax: the CTA's best key per row of A
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(Aux) <= kAuxBytes, "aux area too small");

// k-blocks per stage for one or two column groups: eight products either way
__host__ __device__ constexpr int stage_kblocks(int groups) { return groups == 1 ? 2 : 1; }
__host__ inline int ring_stages(int groups, int block_bytes) {
    const int s = (kSmemLimit - kAuxBytes - kWindowBytes) / (stage_kblocks(groups) * block_bytes);
    return s < kMaxStages ? s : kMaxStages;
}
// (the pad behind the ring: the window of the last stage may reach one window past it)
__host__ inline int smem_bytes(int groups, int stages, int block_bytes) {
    const int used = kAuxBytes + stages * stage_kblocks(groups) * block_bytes + kWindowBytes;
    return used > kSmemAlone ? used : kSmemAlone;
}

// How a product of M rows of A and N rows of B is laid out on `pairs` CTA pairs: the fields of GemmParams that follow from
// the sizes.  Every pair gets the same number of 16-row units of B, cut into as few tiles as the height limit allows.
// Which operand takes the lanes: the one of which a tile has more rows, since an instruction takes as long as it has
// columns.  Measured with rows of B / rows of A on the lanes, us, weights not in L2, tile height h against a group's rows r:
// argmax, K 1024 -> 5000 (h 80) at r 64: 10.5 / 10.8, 112: 11.9 / 10.9, 208: 14.5 / 11.3, 256: 15.5 / 12.5, 2 x 192:
// 20.8 / 17.6; K 2112 -> 32000 (h 224) at r 112: 27.1 / 30.6, 208: 33.0 / 33.2, 256: 35.9 / 33.5, 2 x 192: 51.3 / 57.0.
// Store, 1024 -> 4736 (h 64) at r 48: 19.3 / 19.4, 64: 22.9 / 20.1, 208: 46.4 / 45.4, 2 x 192: 86.9 / 78.0.
__host__ inline bool rows_on_lanes(const GemmParams& g, Epilogue epi) {
    return epi == kEpiStore ? g.h_lo <= g.group_rows : g.h_lo < g.group_rows;
}
__host__ inline int column_groups(int M) { return M <= kGroupRows ? 1 : 2; }
__host__ inline int product_pairs(int N, int sms) { return (N + 15) / 16 < sms / 2 ? (N + 15) / 16 : sms / 2; }
__host__ inline GemmParams product_plan(int M, int N, int K, int pairs) {
    const int groups = column_groups(M);
    GemmParams g{};
    g.M = M; g.N = N; g.K = K;
    g.group_rows = (M + 16 * groups - 1) / (16 * groups) * 16;
    const int units = (N + 15) / 16, per_pair = (units + pairs - 1) / pairs;
    g.rounds = (per_pair + kMaxTile / 16 - 1) / (kMaxTile / 16);
    g.h_lo = per_pair / g.rounds * 16;
    g.tall_rounds = per_pair % g.rounds;
    g.block_bytes = (g.h_lo + (g.tall_rounds ? 16 : 0) + groups * g.group_rows) / 2 * kBK * 2;
    g.stages = ring_stages(groups, g.block_bytes);
    return g;
}

__device__ __forceinline__ uint64_t l2_policy_evict_last() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
// .cta_group::2 form of the tile copy: destination in this CTA, completion counted on `bar_cluster`, a
// shared::cluster address that may lie in the peer CTA.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const void* tmap, uint32_t bar_cluster, int c0, int c1, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
        : : "r"(dst), "l"(tmap), "r"(bar_cluster), "r"(c0), "r"(c1), "l"(policy) : "memory");
}

__device__ __forceinline__ float redux_max_f32(float x) {       // over the warp; NaN drops out
    float y;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(x));
    return y;
}
// The arg-max of 32 columns (rows of A) over a warp's 32 lanes (rows of B, `valid` the mask of those that exist): lane j
// gets column j's key.  NaN reads as -inf.
__device__ __forceinline__ unsigned long long warp_column_argmax(const uint32_t (&v)[32], bool lane_valid, uint32_t valid, uint32_t row0) {
    const int lane = threadIdx.x & 31;
    float best = -INFINITY;
    uint32_t who = 0u;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const float x = lane_valid ? fmaxf(__uint_as_float(v[j]), -INFINITY) : -INFINITY;
        const float m = redux_max_f32(x);
        const uint32_t at = __ballot_sync(0xffffffffu, x == m);
        if (lane == j) { best = m; who = at; }
    }
    return argmax_key(best, row0 + (uint32_t)__ffs((int)(who & valid)) - 1u);          // the lowest row of B among equals
}

// The arg-max of a row's columns [0, count) of 32, this lane's, folded into its best so far; `col0` is the first one's index.
// NaN reads as -inf.  Columns come in ascending order: a later one wins only if it is larger.
__device__ __forceinline__ void lane_row_argmax(const uint32_t (&v)[32], int count, uint32_t col0, float& best, uint32_t& who) {
    float m = -INFINITY;
#pragma unroll
    for (int j = 0; j < 32; ++j)
        if (j < count) m = fmaxf(m, __uint_as_float(v[j]));
    if (who == kNobody || m > best) {
        best = m;
#pragma unroll
        for (int j = 31; j >= 0; --j)
            if (j < count && fmaxf(__uint_as_float(v[j]), -INFINITY) == m) who = col0 + j;
    }
}

// gridDim.x is even: CTAs 2j and 2j + 1 are pair j.
// (kEpiStore: at most 128 registers, so that a CTA of the cell kernel fits beside one: its reads before the wait then lie under
// the product.  With 221 registers / with 128, us per cell call with the weights not in L2: 3 x 2048 -> 5076 23.8 / 23.4, 10 x 4096 ->
// 4096 28.1 / 27.5, 10 x 4096 -> 12288 67.7 / 66.9, 32 x 8192 -> 8192 94.0 / 90.0, 64 x 4096 -> 12288 85.7 / 82.0; runs of one side
// differ by 0.1.)
template <int kEpi, int kGroups, bool kRowsOnLanes>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, kEpi == kEpiStore ? 2 : 1)
gemm_umma_kernel(const GemmParams p, const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap_hi,
                 const __grid_constant__ CUtensorMap bmap_lo) {
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int kQ = stage_kblocks(kGroups);
    constexpr uint32_t kBufs = kGroups == 1 ? 2 : 1;    // accumulator buffers
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t ring = smem_u32(smem) + kAuxBytes;
    const int stages = p.stages, bbytes = p.block_bytes;
    Aux* aux = reinterpret_cast<Aux*>(smem);
    volatile int* abort_flag = &aux->abort_flag;
    const uint32_t rank = cluster_cta_rank();           // 0: issues the products; 1: its peer
    const int pair = (int)(blockIdx.x >> 1), pairs = (int)(gridDim.x >> 1);
    // the peer's abort flag: a wait that gives up here ends the peer's waits too
    const uint32_t peer_abort = cluster_map(smem_u32(&aux->abort_flag), rank ^ 1u);
    auto wait = [&](uint32_t bar, uint32_t parity) {
        const bool ok = mbar_wait_cluster_ns(bar, parity, abort_flag, kWaitLimitNs);
        if (!ok) st_cluster_u32(peer_abort, 1u);
        return ok;
    };
    const bool misaligned = (ring & 1023u) != 0;       // operand tiles must sit on swizzle-atom boundaries (same in both CTAs)
    if (tid == 0) {
        for (int i = 0; i < stages; ++i) { mbar_init(smem_u32(&aux->full[i]), 1); mbar_init(smem_u32(&aux->empty[i]), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&aux->acc_full[i]), 1); mbar_init(smem_u32(&aux->acc_empty[i]), 256); }
        aux->abort_flag = 0;
        fence_barrier_init();
        tma_prefetch_desc(&amap);
        tma_prefetch_desc(&bmap_hi);
        tma_prefetch_desc(&bmap_lo);
    }
    if (kEpi == kEpiArgmax && !kRowsOnLanes)
        for (int i = tid; i < kMaxRows; i += kThreads) aux->best[i] = 0ull;
    if (warp == 0 && !misaligned) { tmem_alloc_pair(smem_u32(&aux->tmem_base), 512); tmem_relinquish_pair(); }
    if (warp == 0 && lane == 0 && !misaligned) {
        // Ask for the ring's first fill of B to be brought to L2 under the tail of whatever precedes this kernel.  That
        // hands nothing to this kernel yet: the copies below read L2, which holds what was written last.
        // (cell 10 x 4096 -> 12288 75.2 -> 72.0 us, 3 x 2048 -> 5076 26.4 -> 25.5, LM head 30 x 2688 -> 32000 33.0 -> 32.2.)
        const CUtensorMap* bmap = p.tall_rounds ? &bmap_hi : &bmap_lo;
        const int share = (p.tall_rounds ? p.h_lo + 16 : p.h_lo) >> 1, row = pair * 2 * share + (int)rank * share;
        const int blocks = min(p.K / kBK, stages * kQ);
        if (row < p.N)
            for (int kb = 0; kb < blocks; ++kb)
                asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" ::"l"(bmap), "r"(kb * kBK), "r"(row) : "memory");
    }
    // may be launched as a programmatic dependent of the kernel before it in the stream: the set-up above touched no
    // input and ran beside that kernel's tail; from here on it has completed (a no-op in an ordinary launch).  The
    // kernel after this one may queue up in turn; before its own wait it reads inputs of the call only (ld_early).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    tc_fence_before();
    cluster_sync_all();            // both CTAs' barriers are initialised and both halves of tensor memory allocated
    tc_fence_after();
    if (misaligned) {
        if (tid == 0) report(p.status, kErrTimeout);
        return;
    }
    const uint32_t tmem = aux->tmem_base;
    const int kblocks = p.K / kBK;
    const int a_half = p.group_rows >> 1;                            // rows of a group of A that this CTA stages
    // round t: one tile per pair, the rounds' bands of B one after the other; a tile that starts past N is empty
    auto tile_rows = [&](int t) { return t < p.tall_rounds ? p.h_lo + 16 : p.h_lo; };
    auto tile_row0 = [&](int t) {
        const int hi = t < p.tall_rounds ? t : p.tall_rounds;
        return pairs * (hi * (p.h_lo + 16) + (t - hi) * p.h_lo) + pair * tile_rows(t);
    };
    const uint32_t full_bar = smem_u32(&aux->full[0]), empty_bar = smem_u32(&aux->empty[0]);
    uint32_t issued = 0;

    if (warp == 0) {
        if (lane == 0) {
            const uint64_t stream_policy = l2_policy_evict_first();   // B is read once
            const uint64_t keep_policy = l2_policy_evict_last();      // A is read by every pair for every tile
            uint32_t stage = 0, ph = 1;
            bool peek = true;                                         // the first pass over the ring finds it empty
            bool going = true;      // nothing is issued any more after a wait that gave up: `issued` counts in ring order
            for (int t = 0; t < p.rounds; ++t) {
                const int row0 = tile_row0(t), share = tile_rows(t) >> 1;
                if (row0 >= p.N) break;
                const CUtensorMap* bmap = t < p.tall_rounds ? &bmap_hi : &bmap_lo;   // box = this CTA's half of the tile's rows
                const int brow = row0 + (int)rank * share, arow = (int)rank * a_half;
                // both CTAs' copies of a stage complete on the even CTA's barrier, which expects all their bytes
                const uint32_t bytes = (uint32_t)(2 * kQ * (share + kGroups * a_half) * kBK * 2);
                for (int kb = 0; kb < kblocks; kb += kQ) {
                    going = going && (peek || wait(empty_bar + stage * 8u, ph));
                    if (going) {
                        const uint32_t full = full_bar + stage * 8u, full0 = cluster_map(full, 0);
                        const uint32_t dst = ring + stage * (uint32_t)(kQ * bbytes);
                        if (rank == 0) mbar_arrive_expect_tx(full, bytes);
#pragma unroll
                        for (int q = 0; q < kQ; ++q) {
                            // (with an odd number of k-blocks the last stage's second one lies past K: the boxes read zeros)
                            const int k0 = (kb + q) * kBK;
                            uint32_t d = dst + q * bbytes;
                            tma_load_2d_pair(d, bmap, full0, k0, brow, stream_policy);
                            d += (uint32_t)share * (kBK * 2);
#pragma unroll
                            for (int g = 0; g < kGroups; ++g)
                                tma_load_2d_pair(d + g * a_half * (kBK * 2), &amap, full0, k0, arow + g * p.group_rows, keep_policy);
                        }
                        ++issued;
                    }
                    if (++stage == (uint32_t)stages) { stage = 0; ph ^= 1u; }
                    peek = mbar_try_wait_cluster(empty_bar + stage * 8u, ph);
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            const uint64_t desc0 = umma_smem_desc_sw128(ring, 16, 1024);     // operands differ in the start address only
            const uint32_t desc_hi = (uint32_t)(desc0 >> 32), desc_lo = (uint32_t)desc0;
            uint32_t stage = 0, ph = 0, tcount = 0;
            bool peek = false;
            for (int t = 0; t < p.rounds; ++t, ++tcount) {
                if (tile_row0(t) >= p.N) break;
                const uint32_t buf = tcount % kBufs, acc_ph = (tcount / kBufs) & 1u;
                const uint32_t a_off = (uint32_t)(tile_rows(t) >> 1) * (kBK * 2) >> 4, a_step = (uint32_t)a_half * (kBK * 2) >> 4;
                const uint32_t d = tmem + buf * 256u;
                const uint32_t idesc = umma_idesc_16bit(256, kRowsOnLanes ? tile_rows(t) : p.group_rows, 0, 0, false);
                bool ok = wait(smem_u32(&aux->acc_empty[buf]), acc_ph ^ 1u);      // both epilogues have read this buffer
                for (int kb = 0; kb < kblocks; kb += kQ) {
                    ok = (peek || wait(full_bar + stage * 8u, ph)) && ok;
                    tc_fence_after();
                    const uint32_t used = empty_bar + stage * 8u;
                    const uint32_t stage_lo = desc_lo + (stage * (uint32_t)(kQ * bbytes) >> 4);
                    if (++stage == (uint32_t)stages) { stage = 0; ph ^= 1u; }
                    if (ok) {
#pragma unroll
                        for (int q = 0; q < kQ; ++q) {
                            const uint32_t b_lo = stage_lo + (uint32_t)(q * bbytes >> 4);
#pragma unroll
                            for (int g = 0; g < kGroups; ++g) {
                                const uint32_t a_lo = b_lo + a_off + g * a_step;
                                const uint32_t lanes_lo = kRowsOnLanes ? a_lo : b_lo, columns_lo = kRowsOnLanes ? b_lo : a_lo;
#pragma unroll
                                for (int ks = 0; ks < kBK / 16; ++ks)    // 32 bytes along K inside the 128-byte swizzle row
                                    umma_ss_pair_lh(d + g * 256u, lanes_lo + ks * 2, desc_hi, columns_lo + ks * 2, desc_hi, idesc,
                                                    (q | ks) ? 1u : (kb ? 1u : 0u));
                            }
                        }
                        umma_commit_pair(used, 3);                       // the slot is free in both CTAs
                    }
                    peek = mbar_try_wait_cluster(full_bar + stage * 8u, ph);
                }
                if (ok) umma_commit_pair(smem_u32(&aux->acc_full[buf]), 3);
            }
        }
    } else if (warp >= 4) {
        const uint32_t lane_sel = (uint32_t)((warp & 3) * 32) << 16;
        const int chunks = (p.group_rows + 31) / 32;
        // kRowsOnLanes: this lane's row of A in each group, and its best so far
        const int my_row = (int)rank * a_half + (warp & 3) * 32 + lane;
        const bool warp_has_rows = (warp & 3) * 32 < a_half, row_on_lane = (warp & 3) * 32 + lane < a_half;
        const bool c_aligned = (reinterpret_cast<uintptr_t>(p.c) & 15) == 0 && (p.ldc & 3) == 0;
        // this call's set of keys (the dependency wait lies before: the walk before this call has moved the number on)
        unsigned long long* row_key = nullptr;
        if (kEpi == kEpiArgmax) {
            const uint32_t call = __ldcg(p.sets.call);
            row_key = p.sets.keys + (size_t)(call & 1u) * p.sets.stride;
            if (blockIdx.x == 0 && tid == 128) p.sets.call[1] = call;
        }
        float best[kGroups];
        uint32_t who[kGroups];
#pragma unroll
        for (int g = 0; g < kGroups; ++g) { best[g] = -INFINITY; who[g] = kNobody; }
        uint32_t tcount = 0;
        for (int t = 0; t < p.rounds; ++t, ++tcount) {
            const int row0 = tile_row0(t);
            if (row0 >= p.N) break;
            const uint32_t buf = tcount % kBufs, acc_ph = (tcount / kBufs) & 1u;
            const int share = tile_rows(t) >> 1;
            // (one verdict for the warp: what follows are warp-wide instructions)
            const bool ok = __all_sync(0xffffffffu, wait(smem_u32(&aux->acc_full[buf]), acc_ph));
            tc_fence_after();
            const int first = row0 + (int)rank * share;                 // this CTA's rows of B: [first, end)
            const int end = first + share < p.N ? first + share : p.N;
            const int warp_row = first + (warp & 3) * 32;               // row of B in the warp's lane 0
            const bool lane_valid = warp_row + lane < end;
            const uint32_t valid = __ballot_sync(0xffffffffu, lane_valid);
            if (kRowsOnLanes) {
                const int cols = min(tile_rows(t), p.N - row0);               // rows of B that exist: the columns here
                if (ok && warp_has_rows) {
#pragma unroll
                    for (int g = 0; g < kGroups; ++g) {
                        const int row = g * p.group_rows + my_row;
#pragma unroll 1
                        for (int c0 = 0; c0 < cols; c0 += 32) {
                            uint32_t v[32];
                            tmem_ld32(tmem + lane_sel + buf * 256u + g * 256u + c0, v);
                            tmem_wait_ld();
                            if (kEpi == kEpiArgmax) {
                                lane_row_argmax(v, cols - c0, (uint32_t)(row0 + c0), best[g], who[g]);
                            } else if (row_on_lane && row < p.M) {
                                float* dst = p.c + (long long)row * p.ldc + row0 + c0;
                                if (c_aligned && cols - c0 >= 32) {
#pragma unroll
                                    for (int j = 0; j < 32; j += 4)
                                        *reinterpret_cast<uint4*>(dst + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                                } else {
#pragma unroll
                                    for (int j = 0; j < 32; ++j)
                                        if (c0 + j < cols) dst[j] = __uint_as_float(v[j]);
                                }
                            }
                        }
                    }
                }
            } else if (ok && warp_row < end) {
#pragma unroll 1
                for (int g = 0; g < kGroups; ++g) {
#pragma unroll 1
                    for (int c4 = 0; c4 < chunks; ++c4) {
                        // (a chunk's columns past the group's rows hold no data of this tile)
                        const int a0 = g * p.group_rows + c4 * 32, left = min(p.M - a0, p.group_rows - c4 * 32);
                        uint32_t v[32];
                        tmem_ld32(tmem + lane_sel + buf * 256u + g * 256u + c4 * 32, v);
                        tmem_wait_ld();
                        if (kEpi == kEpiArgmax) {
                            const unsigned long long key = warp_column_argmax(v, lane_valid, valid, (uint32_t)warp_row);
                            if (lane < left) atomicMax(&aux->best[a0 + lane], key);
                        } else if (lane_valid) {
                            float* dst = p.c + (long long)a0 * p.ldc + warp_row + lane;
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (j < left) dst[j * p.ldc] = __uint_as_float(v[j]);
                        }
                    }
                }
            }
            tc_fence_before();
            // unconditional: the issuing thread's wait on the even CTA's barrier must end
            mbar_arrive_cluster(cluster_map(smem_u32(&aux->acc_empty[buf]), 0));
        }
        if (kEpi == kEpiArgmax && kRowsOnLanes) {
#pragma unroll
            for (int g = 0; g < kGroups; ++g)
                if (row_on_lane && g * p.group_rows + my_row < p.M && who[g] != kNobody)
                    atomicMax(row_key + g * p.group_rows + my_row, argmax_key(best[g], who[g]));
        } else if (kEpi == kEpiArgmax) {
            asm volatile("bar.sync 1, 128;" ::: "memory");              // the four epilogue warps
            for (int i = tid - 128; i < p.M; i += 128)
                if (aux->best[i]) atomicMax(row_key + i, aux->best[i]);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (aux->abort_flag && warp == 0 && lane == 0) {
        if (rank == 0) {
            // both CTAs' copies complete on this CTA's barriers: give those in flight a bounded time to land before
            // either CTA's shared memory is released (the peer leaves only after the cluster barrier below).  The peer's
            // producer may have gone on for longer than this one: the turn past the last is that time for its copies.
            const uint32_t first = issued > (uint32_t)stages ? issued - stages : 0u;
            for (uint32_t it = first; it <= issued; ++it) {
                const uint32_t bar = smem_u32(&aux->full[it % stages]), ph = (it / stages) & 1u;
                for (int polls = 0; polls < (1 << 20) && !mbar_try_wait_cluster(bar, ph); ++polls) {}
            }
        }
        report(p.status, kErrTimeout);
    }
    // no CTA leaves while its peer may still send it an arrival or read or write its half of a product
    __syncthreads();
    cluster_sync_all();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, 512);
    }
}

// Row-major bf16 matrix [rows, K] as a 2-D tensor map with boxes of 64 columns x box_rows rows (128-byte swizzle; a
// multiple of 8 rows up to 256): one box is one operand tile in the canonical K-major layout.  Rows past the end read
// as zeros.
inline int make_operand_map(EncodeTiledFn encode, CUtensorMap* map, const void* ptr, long long rows, long long K, int box_rows) {
    if (!encode) return -1;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
    const cuuint32_t box[2] = {kBK, (cuuint32_t)box_rows};
    const cuuint32_t elem_strides[2] = {1, 1};
    return (int)encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, elem_strides,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

}  // namespace gemm_path

// ------------------------------------------------------------------------------------------------------------
// The drafter cell's element-wise half (Eq. 2, 5-8) over the fp32 pre-activations
// S = h [W^f; W^i; W^o; W^c]^T ([rows, 4d]).  f = layer normalisation (biased variance, eps inside the root,
// optional affine) followed by exact GeLU.
// A row is spread over a cluster of 8 CTAs (a handful of rows would otherwise sit on a handful of SMs: 10 rows of
// 12288 took 30 us on one CTA each).  The statistics of the two layer normalisations are over the whole row: one
// exchange through distributed shared memory and one cluster barrier each (cluster_mean_rstd).
// ------------------------------------------------------------------------------------------------------------
constexpr int kCellCluster = 8;
constexpr int kCellThreads = 512;
constexpr int kCellPerThread = 4;                // d <= 8 * 512 * 4 = 16384
constexpr int kCellMaxD = kCellCluster * kCellThreads * kCellPerThread;

struct CellParams {
    const float* s;                  // [rows, 4d]: W^f h, W^i h, W^o h, W^c h
    const __nv_bfloat16* emb;        // [rows, d]  E(t), Eq. 1
    const float* gamma_c; const float* beta_c;   // affine of f in Eq. 6 (may be null)
    const float* gamma_z; const float* beta_z;   // affine of f in Eq. 8 (may be null)
    float* z;                        // [rows, d] in / out
    float* h_f32;                    // [rows, d] out (may be null)
    __nv_bfloat16* h_bf16;           // [rows, d] out (may be null)
    int d;
    float alpha, eps;
};

constexpr int kCellWarps = kCellThreads / 32;
struct CellStats { float2 warp[kCellWarps], cta[kCellCluster]; };      // (mean, sum of squared deviations) of a warp's, a CTA's columns

template <int kLanes>
__device__ __forceinline__ float cell_lanes_sum(float v) {
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// Columns of a CTA with `count` of them that warp w holds.
__device__ __forceinline__ int cell_warp_columns(int count, int w) {
    int n = 0;
#pragma unroll
    for (int k = 0; k < kCellPerThread; ++k) n += min(max(count - k * kCellThreads - w * 32, 0), 32);
    return n;
}
// Mean and sum of squared deviations of kLanes sets of n columns each, one per lane (the same in every group of kLanes), by the
// pairwise-variance identity  M2 = sum_i M2_i + sum_i n_i (mean_i - mean)^2 : no cancellation.
template <int kLanes>
__device__ __forceinline__ float2 cell_combine(float2 pair, float n, float total) {
    const float mean = cell_lanes_sum<kLanes>(n * pair.x) / fmaxf(total, 1.f), dm = pair.x - mean;
    return make_float2(mean, cell_lanes_sum<kLanes>(pair.y + n * dm * dm));
}

// Mean and 1 / sqrt(variance + eps) over a whole row from the values x[] this thread holds (on[] says which exist).
// Each warp takes the pair of its own columns, the first one combines them and pushes the CTA's into every CTA of the cluster,
// and after one cluster barrier every warp combines the eight: the same numbers everywhere, and nobody reads a peer's shared
// memory after the barrier.  (With every warp's pair pushed and 128 of them combined by every warp, us per call: 384 x 1024 -> 4096
// 97.6, now 89.0; 200 x 2048 -> 2048 53.5, now 48.3; 10 x 4096 -> 4096 27.7, now 27.5.  With two block sums, four CTA barriers,
// before the exchange instead of one: 96.6, 52.3, 29.8.)
__device__ __forceinline__ void cluster_mean_rstd(const float (&x)[kCellPerThread], const bool (&on)[kCellPerThread], int count,
                                                  int slice, int d, float eps, CellStats& stats, float& mean, float& rstd) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < kCellPerThread; ++k) sum += on[k] ? x[k] : 0.f;
    const int n_warp = cell_warp_columns(count, warp);
    const float mean_warp = cell_lanes_sum<32>(sum) / (float)max(n_warp, 1);
    float sq = 0.f;
#pragma unroll
    for (int k = 0; k < kCellPerThread; ++k)
        if (on[k]) { const float t = x[k] - mean_warp; sq += t * t; }
    const float m2_warp = cell_lanes_sum<32>(sq);
    if (lane == 0) stats.warp[warp] = make_float2(mean_warp, m2_warp);
    __syncthreads();
    if (warp == 0) {
        const int w = lane % kCellWarps;
        const float2 cta = cell_combine<kCellWarps>(stats.warp[w], (float)cell_warp_columns(count, w), (float)count);
        if (lane < kCellCluster) cluster.map_shared_rank(&stats, lane)->cta[cluster.block_rank()] = cta;
    }
    cluster.sync();
    const int r = lane % kCellCluster;
    const float2 row = cell_combine<kCellCluster>(stats.cta[r], (float)min(slice, max(d - r * slice, 0)), (float)d);
    mean = row.x;
    rstd = rsqrtf(row.y / d + eps);
}

__device__ __forceinline__ float gelu_exact(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float sigmoid_f(float x) { return 1.f / (1.f + __expf(-x)); }

__global__ void __cluster_dims__(kCellCluster, 1, 1) __launch_bounds__(kCellThreads, 2) lstm_cell_kernel(const CellParams p) {
    namespace cg = cooperative_groups;
    __shared__ CellStats s_stats[2];                 // of the two normalisations
    cg::cluster_group cluster = cg::this_cluster();
    const long long row = blockIdx.x / kCellCluster;
    const int d = p.d;
    const int slice = (d + kCellCluster - 1) / kCellCluster;
    const int j0 = (int)cluster.block_rank() * slice;             // this CTA's columns: [j0, min(j0 + slice, d))
    const int count = min(slice, max(d - j0, 0));
    const float* s = p.s + row * 4ll * d;
    // Every CTA of the cluster is running before anyone writes into its shared memory: they tell each other so here and look
    // when all loads are on their way.  (A whole barrier here put S behind it, in every wave of many rows: 384 x 1024 -> 4096 99.4 us
    // instead of 97.5, 200 x 2048 -> 2048 54.7 instead of 53.5.)
    cluster.barrier_arrive();
    // A programmatic dependent of the product, which writes S and nothing else: E(t), z and the affine parameters are read
    // (ld_early) under the product's tail.
    float xc[kCellPerThread], sf[kCellPerThread], si[kCellPerThread], so[kCellPerThread], zo[kCellPerThread], zn[kCellPerThread];
    float ae[kCellPerThread], gc[kCellPerThread], bc[kCellPerThread];
    bool on[kCellPerThread];
#pragma unroll
    for (int k = 0; k < kCellPerThread; ++k) {
        const int i = k * kCellThreads + threadIdx.x, j = j0 + i;
        on[k] = i < count;
        xc[k] = sf[k] = si[k] = so[k] = zo[k] = zn[k] = ae[k] = bc[k] = 0.f;
        gc[k] = 1.f;
        if (on[k]) {
            ae[k] = p.alpha * __bfloat162float(ld_early(p.emb + row * d + j));
            zo[k] = ld_early(p.z + row * d + j);
            if (p.gamma_c) gc[k] = ld_early(p.gamma_c + j);
            if (p.beta_c) bc[k] = ld_early(p.beta_c + j);
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");      // the kernel after this one may queue up
#pragma unroll
    for (int k = 0; k < kCellPerThread; ++k) {
        const int j = j0 + k * kCellThreads + threadIdx.x;
        if (on[k]) {     // s^m = W^m h + alpha e  (Eq. 2)
            xc[k] = __ldcg(s + 3ll * d + j) + ae[k]; sf[k] = __ldcg(s + j) + ae[k];
            si[k] = __ldcg(s + 1ll * d + j) + ae[k]; so[k] = __ldcg(s + 2ll * d + j) + ae[k];
        }
    }
    cluster.barrier_wait();
    float mean_c, rstd_c;
    cluster_mean_rstd(xc, on, count, slice, d, p.eps, s_stats[0], mean_c, rstd_c);
    // z' = z g^f + f(s^c) g^i  (Eq. 5-7)
#pragma unroll
    for (int k = 0; k < kCellPerThread; ++k) {
        const int j = j0 + k * kCellThreads + threadIdx.x;
        if (on[k]) {
            const float y = (xc[k] - mean_c) * rstd_c * gc[k] + bc[k];
            zn[k] = zo[k] * sigmoid_f(sf[k]) + gelu_exact(y) * sigmoid_f(si[k]);
            p.z[row * d + j] = zn[k];
        }
    }
    // (asked for here, to arrive under the second exchange: read before the wait with the others they made the kernel spill 40
    // bytes; 64 x 4096 -> 12288 85.5 -> 84.0 us per call, 32 x 8192 -> 8192 91.2 -> 90.6, 10 x 4096 -> 12288 67.6 -> 67.2)
    float gz[kCellPerThread], bz[kCellPerThread];
#pragma unroll
    for (int k = 0; k < kCellPerThread; ++k) {
        const int j = j0 + k * kCellThreads + threadIdx.x;
        gz[k] = on[k] && p.gamma_z ? __ldcg(p.gamma_z + j) : 1.f;
        bz[k] = on[k] && p.beta_z ? __ldcg(p.beta_z + j) : 0.f;
    }
    float mean_z, rstd_z;
    cluster_mean_rstd(zn, on, count, slice, d, p.eps, s_stats[1], mean_z, rstd_z);
    // h' = f(z') g^o  (Eq. 8)
#pragma unroll
    for (int k = 0; k < kCellPerThread; ++k) {
        const int j = j0 + k * kCellThreads + threadIdx.x;
        if (on[k]) {
            const float y = (zn[k] - mean_z) * rstd_z * gz[k] + bz[k];
            const float h = gelu_exact(y) * sigmoid_f(so[k]);
            if (p.h_f32) p.h_f32[row * d + j] = h;
            if (p.h_bf16) p.h_bf16[row * d + j] = __float2bfloat16_rn(h);
        }
    }
}

}  // namespace owl
