// LSE merge of the split-KV partials: for every output row whose keys were processed by more than
// one CTA, out = sum_s exp(lse_s - lse) o_s with lse = ln sum_s exp(lse_s); rounded to bf16.
#pragma once

#include <cuda_fp16.h>

#include "owl_common.cuh"
#include "accept.cuh"

namespace owl {

constexpr int kCombineWarps = 8;
constexpr int kCombineThreads = (kCombineWarps + 1) * 32;     // and one that rehearses
constexpr int kRehearsedPartials = 5;                         // the unrolled loops and what they leave over
constexpr int kCombineCtasPerSm = 4;
constexpr int kCombineRows = 8;            // a unit's rows that a CTA merges at a time

// Partials per round of the merge, for `units` units (sequence, KV head) cut by `ctas` CTAs: as many as a unit of
// average length is cut into, plus one at either end, so that its rows take one memory round trip; longer units take
// several rounds.  A stage of 32 rows for everybody made a CTA 128 KB large: one per SM, and the 1920 rows of a 60-node
// tree (240 CTAs) ran in two waves.
inline int combine_group(long long units, int ctas) {
    const long long g = (ctas + units - 1) / units + 2;
    return (int)(g < 4 ? 4 : g < 32 ? g : 32);
}
__host__ __device__ inline int rehearsed_partials(int group) { return group < kRehearsedPartials ? group : kRehearsedPartials; }
inline size_t combine_stage_bytes(int group, int lg_parts) {
    return (size_t)((kCombineWarps >> lg_parts) * group + rehearsed_partials(group)) * 34 * sizeof(float4);
}
inline int combine_ctas_per_sm(int group) {
    const int fit = (int)((227u << 10) / (combine_stage_bytes(group, 0) + 1024));
    return fit < kCombineCtasPerSm ? fit : kCombineCtasPerSm;
}
// CTAs that share a block's channels: 1, 2 or 4, as long as every one still has an SM to itself.  What a merge waits for is
// the partials that one SM takes in and folds, 70 KB for the eight rows of a block at 2K context (chain of 8 nodes: 32 blocks on 128 SMs
// instead of 32, and the schedule's shorter divisions, 12.1 -> 11.5 us per step).
inline int combine_lg_parts(long long blocks, int other_ctas, int sms) {
    int lg = 0;
    while (lg < 2 && (blocks << (lg + 1)) + other_ctas <= sms) ++lg;
    return lg;
}
// What a launch of `ctas` CTAs asks for: its stage, and enough that no SM takes more than its share of them.  The
// SMs whose attention CTA ends first would otherwise collect several merge CTAs each (2K context, 33 CTAs: 15.5 -> 16.1 us
// per step).
inline size_t combine_smem_bytes(int group, int lg_parts, unsigned ctas, int sms) {
    const unsigned share = (ctas + (unsigned)sms - 1) / (unsigned)sms;
    const size_t spread = (227u << 10) / (share + 1) + 16, stage = combine_stage_bytes(group, lg_parts);
    return stage > spread ? stage : spread;
}

// Blocks of eight rows that hold any, of all units of a sequence with n nodes.
__host__ __device__ inline int seq_blocks(int n, int group, int num_kv_heads) {
    return num_kv_heads * ((n * group + kCombineRows - 1) / kCombineRows);
}
// At most so many in a call: the host knows the nodes of the batch and the most that a sequence has.
inline long long combine_most_blocks(long long batch, long long total_nodes, int max_nodes, int group, int num_kv_heads) {
    const long long by_max = batch * seq_blocks(max_nodes, group, 1), by_total = (total_nodes * group + (kCombineRows - 1) * batch) / kCombineRows;
    return num_kv_heads * (by_max < by_total ? by_max : by_total);
}

// Lines that are not short: what the merge goes by, whichever are fewer, the units or the places where the line of a pass of
// `ctas` CTAs is cut (one CTA: none, but a grid is never empty).
__host__ __device__ inline int combine_cuts(int ctas) { return ctas > 1 ? ctas - 1 : 1; }
__host__ __device__ inline int combine_places(int units, int ctas) { return units < combine_cuts(ctas) ? units : combine_cuts(ctas); }
// CTAs per place: one for each block of the largest unit there may be, while all are resident at once.
inline int combine_turns(int group, int max_nodes, int places, long long most_ctas) {
    const long long blocks = seq_blocks(max_nodes, group, 1), most = most_ctas / places;
    return (int)(blocks < most ? blocks : most > 1 ? most : 1);
}
// The unit whose tiles are cut at t, a piece's first place, which lies in the sequence [begin, end) of the line: its KV head and
// its length with the gap.  False: the piece begins with a unit, or in the gap before one.
__host__ __device__ inline bool cut_unit(const Partition<long long>& part, long long t, long long begin, long long end, int kv_heads,
                                         int& h, int& len) {
    len = (int)((unsigned)(end - begin) / (unsigned)kv_heads);
    h = (int)((unsigned)(t - begin) / (unsigned)len);
    return (int)(t - begin) - h * len > part.pen;
}
// What a CTA takes of a unit that lies in pieces c0 .. c0 + count - 1: its cuts share its blocks, `turns` CTAs each.
__host__ __device__ inline void cut_share(int cut, int c0, int count, int turn, int turns, int& first, int& stride) {
    first = (cut - c0 - 1) * turns + turn;
    stride = (count - 1) * turns;
}

// Short lines: which block is whose.  Lane b holds sequence b, everything is derived from the inputs; a sequence that the pass
// refuses has no blocks.  (Numbered for every sequence up to the largest tree's rows, the blocks of one tree of 64 nodes among
// chains lay mostly empty and the full ones far apart, two and more to a CTA.  One such tree among 16 sequences of 100-1500
// tokens: 31.2 us per step, now 27.6; among 8 of 200-6000: 46.8, now 44.8.)
struct BlockNumbers {
    int blocks, end;                 // of the call; where this lane's sequence ends
    __device__ __forceinline__ void derive(const AttnParams& p, const WarpSchedule& ws) {
        const int lane = threadIdx.x & 31;
        end = ws.tiles > 0 ? seq_blocks(ws.n, p.group, p.num_kv_heads) : 0;
        for (int o = 1; o < p.batch; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += v;
        }
        blocks = __shfl_sync(0xffffffffu, end, p.batch - 1);
    }
};

// A block of eight of a unit's packed rows per CTA and turn, 16 of the 128 channels per warp: lane = (row, four
// channels).  The warp finds the CTAs whose pieces cut the unit and merges their partials in CTA order.  A CTA stores at
// most two partials: slot 2c if its piece starts inside the unit, else 2c + 1.
//
// Partials lie as the attention kernel's lanes, one row each, can store them straight from registers in whole lines:
// [slot][32 groups of four channels][256 rows][4].  Eight neighbouring rows are then a line of 128 bytes here too.
// (With the rows of a partial one after the other the pass had to turn every 32 x 32 piece over in shared memory: its
// epilogue took 1.9 us instead of 1.0 at 2K context, 3.5 instead of 3.0 for 240 rows at 47K.)
//
// The kernel is launched as a programmatic dependent of that pass and its time after the pass has ended is pure
// latency, so everything that needs no output of the pass comes before the wait: on short lines (small_schedule) the
// warp derives the schedule from the inputs exactly as the pass did (warp_schedule) and knows its
// block's partial slots when the wait returns; what is left is one round of loads.  Otherwise (kManySeqs) it reads the
// schedule the pass left in global memory (first place of every sequence, totals, choice of partition).
//
// kFused (verify step): the grid has one more CTA per sequence after the row CTAs; each of those runs one
// sequence's acceptance walk over the arg-max keys that the pass's spare warps left (`ap`).
//
// p.combine_group: partials fetched per round, at most 32 (combine_group above).  A round's rows go through a
// warp-private stage in shared memory of that many pieces, which is what limits the CTAs per SM.
//
// The stage is there for the sake of the code's length, not of the data: with the pieces in registers the fetch and
// the fold were two loops unrolled 32 times, some 450 instructions that a warp executes once per block, mostly once in
// all, at the pace of instruction fetches from L2.
template <bool kFused, bool kManySeqs>
__global__ void __launch_bounds__(kCombineThreads, kCombineCtasPerSm) combine_sched_kernel(const AttnParams p, const AcceptParams ap) {
    const unsigned row_ctas = (unsigned)p.combine_row_ctas;
    if (kFused) {
        if (blockIdx.x >= row_ctas) {
            static_assert(kCombineThreads >= kArgmaxThreads, "the walk's block");
            if (threadIdx.x < kArgmaxThreads)
                accept_walk_seq(ap, (int)(blockIdx.x - row_ctas), [&] {
                    wait_and_let_dependents_start();
                    return (const unsigned long long*)ap.part_keys;
                });
            return;
        }
    }
    // The row CTAs are persistent (one CTA per eight rows cost a launch of 8192 rows 19 us, most of it the schedule derived
    // 8192 times).  Short lines: a warp derives the schedule once and then takes blocks first, first + stride, ..., numbered
    // sequence by sequence, unit by unit, and only those that hold rows (BlockNumbers).  Otherwise the units are many, and only
    // those that a piece's end cuts have anything to merge: a CTA goes by one cut and takes its share of that unit's blocks; or,
    // where the units are fewer than the cuts, by one unit (one KV head, 40 sequences of 50-2000 tokens with 80 rows: 17.7 us
    // per call, by cuts 21.2; with 256 rows 28.7, by cuts 33.8).  (Every block of every unit looked up in turn, us per step: 64
    // sequences of 100-1500 tokens with one tree of 64 nodes 91.4, now 79.5; 300 of 50-300 tokens 124.4, now 120.1; 1000 of
    // 20-200 with one such tree 540, now 355.)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // The ninth warp rehearses: it runs the code that follows the wait on whatever the first slots hold (out_row stays -1, so
    // nothing is written), while the others derive the schedule and wait.  That code runs once or twice per launch, and its lines
    // used to be fetched when the partials were there already (2.9 -> 2.5 us after the wait; 2K step 12.4 -> 12.1 with the walk's
    // reads before its wait).
    const bool rehearsal = warp == kCombineWarps;
    // A block is shared out to 1 << combine_lg_parts CTAs, each with a part of the channels and of the eight warps.
    const int warps = kCombineWarps >> p.combine_lg_parts, part_no = (int)blockIdx.x & ((1 << p.combine_lg_parts) - 1);
    if (!rehearsal && warp >= warps) return;
    const int r = lane & 7, chunk = rehearsal ? lane >> 3 : (part_no * warps + warp) * 4 + (lane >> 3);   // row of the block; four channels
    extern __shared__ float4 combine_stage[];          // per warp: [group][32] pieces of the partials, [group][8] LSEs
    const int group = rehearsal ? rehearsed_partials(p.combine_group) : p.combine_group;
    float4* stage = combine_stage + (rehearsal ? warps : warp) * p.combine_group * 34;
    float* lse_stage = reinterpret_cast<float*>(stage + group * 32);
    const uint32_t stage_u32 = (uint32_t)__cvta_generic_to_shared(stage + lane);
    // The unit: its sequence's nodes and their offset, its KV head; the first partial's slot and the number of partials (0:
    // nothing to merge).  The block: its first row, this lane's row of the output (-1: past the unit's last).
    int n = 0, node_base = 0, h = 0, slot = 0, count = 0, row0 = 0;
    long long out_row = -1;
    int c0 = 0;
    auto plan = [&](auto t0, int tiles, const auto& part) {       // the unit's place on the line and its tiles
        count = 0;
        // the CTAs that hold its first tile, its last one and, if it is not the line's first, the place before its gap: three
        // lanes find one each
        auto place = t0 + part.pen;
        if (lane == 1) place += tiles - 1;
        if (lane == 2) place = t0 > 0 ? t0 - 1 : 0;
        const int mine = part.owner(place);
        c0 = __shfl_sync(0xffffffffu, mine, 0);
        const int c1 = __shfl_sync(0xffffffffu, mine, 1), before = __shfl_sync(0xffffffffu, mine, 2);
        if (c0 == c1) return;              // a single CTA saw every key of this unit and wrote the result itself
        // the unit's first CTA may have come from another unit or from the gap before that; the others' pieces start in this one
        slot = 2 * c0 + (t0 > 0 && before == c0 ? 1 : 0);
        count = c1 - c0 + 1;
    };
    auto take_rows = [&](int block) {      // of the unit
        row0 = block * kCombineRows;
        const int row = row0 + r, node = (int)row_node(p, row);
        out_row = row < n * p.group ? (long long)(node_base + node) * p.num_q_heads + h * p.group + (row - node * p.group) : -1;
    };
    WarpSchedule ws{};
    BlockNumbers num{};
    auto locate = [&](int id) {            // every lane of the warp, same block
        const int b = __ffs(__ballot_sync(0xffffffffu, id < num.end)) - 1;
        n = __shfl_sync(0xffffffffu, ws.n, b);
        node_base = __shfl_sync(0xffffffffu, ws.node_base, b);
        const int tiles = __shfl_sync(0xffffffffu, ws.tiles, b), unit_blocks = seq_blocks(n, p.group, 1);
        const int local = id - __shfl_sync(0xffffffffu, num.end, b) + p.num_kv_heads * unit_blocks;
        h = div_small(local, unit_blocks);
        take_rows(local - h * unit_blocks);
        plan(__shfl_sync(0xffffffffu, ws.begin, b) + h * (tiles + ws.part.pen), tiles, ws.part);
    };
    // Block numbers are the call's for short lines, the unit's otherwise.
    int id = (int)blockIdx.x >> p.combine_lg_parts, stride = (int)row_ctas >> p.combine_lg_parts, end = 1;
    // latency after the pass has ended is what this kernel costs: whatever needs no output of the pass comes before
    // the wait - for short lines the whole plan of the first block
    if (rehearsal) {
        count = min(kRehearsedPartials, p.num_ctas);
        id = 0;
    } else {
        if (!kManySeqs) {
            ws = warp_schedule(p);
            num.derive(p, ws);
            end = num.blocks;
            if (id < end) locate(id);
        }
        // from here on the split-KV pass has completed and its writes are visible (a no-op in an ordinary launch)
        wait_and_let_dependents_start();
        if (kManySeqs) {
            const int units = p.batch * p.num_kv_heads, places = combine_places(units, p.num_ctas), turns = div_small((int)row_ctas, places);
            const int turn = div_small(id, places), place = id - turn * places;
            const long long* seq_begin = p.sched_seq_begin;
            const SchedHeader* header = p.sched_header;
            Partition<long long> part;
            auto read_partition = [&] {
                const SchedHeader hdr = *header;
                part.init(hdr.total_tiles, p.num_ctas, hdr.units, hdr.uniform_tiles);
            };
            if (places == units) {
                const int b = div_small(place, p.num_kv_heads);
                const long long from = seq_begin[b], to = seq_begin[b + 1];
                n = seq_nodes(p, b);
                node_base = seq_node_base(p, b);
                read_partition();
                const int len = (int)((unsigned)(to - from) / (unsigned)p.num_kv_heads);
                if (len == 0) return;                          // a sequence that the pass refuses
                h = place - b * p.num_kv_heads;
                plan(from + (long long)h * len, len - part.pen, part);
                id = turn;
                stride = turns;
            } else {
                // the first place of piece `cut`: which sequence it lies in, 32 of them at a look, the first look's loads beside the
                // header's
                const int cut = place + 1;
                long long from = 0, to = 0, t, t_end;
                const int per = p.batch > 32 ? 32 : 1, at = lane * per;
                if (at < p.batch) from = seq_begin[at];
                read_partition();
                part.range(cut, t, t_end);
                if (t >= part.total) return;
                const int last = 31 - __clz((int)__ballot_sync(0xffffffffu, at < p.batch && from <= t));
                const int mine = (per > 1 ? last * per : 0) + lane;
                if (mine < p.batch) {
                    from = seq_begin[mine];
                    to = seq_begin[mine + 1];
                    n = seq_nodes(p, mine);
                    node_base = seq_node_base(p, mine);
                }
                const int who = 31 - __clz((int)__ballot_sync(0xffffffffu, mine < p.batch && from <= t));
                n = __shfl_sync(0xffffffffu, n, who);
                node_base = __shfl_sync(0xffffffffu, node_base, who);
                from = __shfl_sync(0xffffffffu, from, who);
                int len;
                if (!cut_unit(part, t, from, __shfl_sync(0xffffffffu, to, who), p.num_kv_heads, h, len)) return;
                plan(from + (long long)h * len, len - part.pen, part);
                cut_share(cut, c0, count, turn, turns, id, stride);
            }
            end = seq_blocks(n, p.group, 1);
        }
    }
    for (bool first = true; id < end; id += stride, first = false) {
        if (kManySeqs) { if (!rehearsal) take_rows(id); }
        else if (!first) locate(id);
        if (count == 0) continue;
        // Partials are taken `group` at a time, their LSEs with them: one memory round trip per group.  Groups are folded
        // online (running maximum, each lane its own row's).
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        float sum = 0.f, mx = -INFINITY;
        bool bad = false;
        // slots of neighbouring CTAs lie two apart; only the first CTA's partial may be its second
        const float4* src = reinterpret_cast<const float4*>(p.part_o) + (slot * 32ll + chunk) * kMaxRows + row0 + r;
        int step = slot & 1 ? 32 * kMaxRows : 64 * kMaxRows;
        for (int base = 0; base < count; base += group) {
            const int cnt = count - base < group ? count - base : group;
            __syncwarp();                                // the stage's weights of the round or the block before have been read
            for (int j = lane; j < 2 * cnt; j += 32) {   // eight rows' LSEs: two pieces of 16 bytes
                const int at = base + (j >> 1), sl = at == 0 ? slot : (slot & ~1) + 2 * at;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(lse_stage + j * 4)),
                             "l"(p.part_lse + (long long)sl * kMaxRows + row0 + (j & 1) * 4) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll 4
            for (int j = 0; j < cnt; ++j) {
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(stage_u32 + (uint32_t)j * 512u), "l"(src) : "memory");
                src += step;
                step = 64 * kMaxRows;
            }
            asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 1;" ::: "memory");
            __syncwarp();
            // the row's four lanes share its weights out, which take the place of the LSEs
            float mx_new = mx;
            for (int j = lane >> 3; j < cnt; j += 4) {
                const float l = lse_stage[j * 8 + r];
                bad = bad || (out_row >= 0 && __float_as_uint(l) == kBadPartial);
                mx_new = fmaxf(mx_new, l);
            }
            mx_new = fmaxf(mx_new, __shfl_xor_sync(0xffffffffu, mx_new, 8));
            mx_new = fmaxf(mx_new, __shfl_xor_sync(0xffffffffu, mx_new, 16));
            float round_sum = 0.f;
            for (int j = lane >> 3; j < cnt; j += 4) {
                const float l = lse_stage[j * 8 + r], w = l > -INFINITY ? __expf(l - mx_new) : 0.f;     // an empty partial has no weight
                lse_stage[j * 8 + r] = w;
                round_sum += w;
            }
            round_sum += __shfl_xor_sync(0xffffffffu, round_sum, 8);
            round_sum += __shfl_xor_sync(0xffffffffu, round_sum, 16);
            const float rescale = mx > -INFINITY ? __expf(mx - mx_new) : 0.f;
            acc.x *= rescale; acc.y *= rescale; acc.z *= rescale; acc.w *= rescale;
            sum = sum * rescale + round_sum;
            mx = mx_new;
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
#pragma unroll 4
            for (int j = 0; j < cnt; ++j) {
                const float w = lse_stage[j * 8 + r];
                const float4 v = stage[j * 32 + lane];             // this lane's own copy
                acc.x += w * v.x; acc.y += w * v.y; acc.z += w * v.z; acc.w += w * v.w;
            }
        }
        const float inv = sum > 0.f ? 1.f / sum : 0.f;
        uint2 pk;
        if (p.f16) {
            __half2 lo2 = __floats2half2_rn(acc.x * inv, acc.y * inv), hi2 = __floats2half2_rn(acc.z * inv, acc.w * inv);
            pk.x = *reinterpret_cast<uint32_t*>(&lo2);
            pk.y = *reinterpret_cast<uint32_t*>(&hi2);
        } else {
            __nv_bfloat162 lo2 = __floats2bfloat162_rn(acc.x * inv, acc.y * inv), hi2 = __floats2bfloat162_rn(acc.z * inv, acc.w * inv);
            pk.x = *reinterpret_cast<uint32_t*>(&lo2);
            pk.y = *reinterpret_cast<uint32_t*>(&hi2);
        }
        const float lse = sum > 0.f ? mx + logf(sum) : -INFINITY;
        // rows past the unit's last hold nothing; a bad tree or page in the unit's sequence (the same for all of its rows): no
        // output
        if (!__any_sync(0xffffffffu, bad) && out_row >= 0) {
            *reinterpret_cast<uint2*>(p.out + out_row * kHeadDim + chunk * 4) = pk;
            if (p.lse && chunk == 0) p.lse[out_row] = lse;
        }
    }
}

}  // namespace owl
