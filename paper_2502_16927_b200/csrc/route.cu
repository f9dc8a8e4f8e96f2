// Routing kernels: per-token top-k with softmax gate values, and the deterministic stable counting
// sort of routed slots by expert that lays out the dropless dispatch (the on-device stand-in for the
// send layout of the first All-to-All).
#include "internal.h"

namespace bigmac {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kNoExpert = 0x7fffffff;          // "no candidate yet" in the arg-max rounds; never written out

// One warp per token.  Lane l holds experts l, l+32, ...  k rounds of warp arg-max under the order
// (logit descending, expert id ascending); gate values are the softmax over the k winners.
// KREG: k <= 32, the j-th winner stays in a register of lane j until one coalesced store at the end; otherwise
// the winners pass through the output arrays.
// Non-finite logits: NaN is ordered as -inf, and a round that finds only -inf among the experts not yet chosen takes
// the lowest such id, so every id written lies in [0, E) whatever the logits hold (k <= E).  A token whose kept
// logits are all -inf gets the gate value 1/k on each.
template <int VPL, bool KREG>
__global__ void __launch_bounds__(256) topk_kernel(const float* __restrict__ logits, const float* __restrict__ b_gate,
                                                   int T, int E, int k, int32_t* __restrict__ topk_idx,
                                                   float* __restrict__ topk_w) {
    grid_dependency_wait();
    grid_dependency_launch();
    const int lane = threadIdx.x & 31;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= T) return;
    const float* row = logits + (size_t)t * E;
    float v[VPL];
#pragma unroll
    for (int i = 0; i < VPL; ++i) {
        const int e = lane + 32 * i;
        const float x = e < E ? row[e] + (b_gate ? b_gate[e] : 0.0f) : -INFINITY;
        v[i] = x == x ? x : -INFINITY;             // NaN is ordered as -inf
    }
    int32_t* out_idx = topk_idx + (size_t)t * k;
    float* out_w = topk_w + (size_t)t * k;
    float my_v = -INFINITY;
    int my_e = 0;
    uint32_t taken = 0;                            // bit i: expert lane + 32 i already chosen
    for (int j = 0; j < k; ++j) {
        float best = -INFINITY;
        int best_e = kNoExpert;
#pragma unroll
        for (int i = 0; i < VPL; ++i) {            // ascending expert id within the lane: strict > keeps the lowest id
            const int e = lane + 32 * i;
            if (e < E && !((taken >> i) & 1u) && (best_e == kNoExpert || v[i] > best)) { best = v[i]; best_e = e; }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const float ov = __shfl_xor_sync(kFull, best, off);
            const int oe = __shfl_xor_sync(kFull, best_e, off);
            if (ov > best || (ov == best && oe < best_e)) { best = ov; best_e = oe; }
        }
        if (best_e != kNoExpert && (best_e & 31) == lane) taken |= 1u << (best_e >> 5);
        if (KREG) {
            if (lane == j) { my_v = best; my_e = best_e; }
        } else if (lane == 0) {
            out_idx[j] = best_e;
            out_w[j] = best;                       // raw logit for now
        }
    }
    if (KREG) {
        const float top = __shfl_sync(kFull, my_v, 0);
        const float ex = lane < k ? (top == -INFINITY ? 1.0f : expf(my_v - top)) : 0.0f;
        float part = ex;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(kFull, part, off);
        if (lane < k) {
            out_idx[lane] = my_e;
            out_w[lane] = ex / part;
        }
        return;
    }
    __syncwarp();
    const float top = out_w[0];
    const bool none = top == -INFINITY;
    float part = 0.0f;
    for (int j = lane; j < k; j += 32) part += none ? 1.0f : expf(out_w[j] - top);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(kFull, part, off);
    for (int j = lane; j < k; j += 32) out_w[j] = (none ? 1.0f : expf(out_w[j] - top)) / part;
}

// Pass 1 of the counting sort.  Block b owns slots [b*kSortChunk, (b+1)*kSortChunk); it writes, per
// slot, the number of earlier slots of the same block routed to the same expert, and per expert the
// block's count.  Warps own consecutive sub-chunks, so the order is the slot order.
__global__ void __launch_bounds__(256) sort_local_kernel(const int32_t* __restrict__ topk_idx, int64_t N, int E,
                                                         int32_t* __restrict__ local_rank,
                                                         int32_t* __restrict__ block_counts) {
    grid_dependency_wait();
    grid_dependency_launch();
    extern __shared__ int32_t warp_run[];            // [8][E]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < 8 * E; i += blockDim.x) warp_run[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortChunk + warp * (kSortChunk / 8);
    int32_t my_rank[kSortChunk / 256];
#pragma unroll
    for (int it = 0; it < kSortChunk / 256; ++it) {
        const int64_t s = base + it * 32 + lane;
        int e = s < N ? topk_idx[s] : -1;
        if ((unsigned)e >= (unsigned)E) e = -1;      // an id outside [0, E) (never written by the top-k kernels) counts nowhere
        const unsigned peers = __match_any_sync(kFull, e);
        const int leader = __ffs(peers) - 1;
        int old = 0;
        if (lane == leader && e >= 0) {
            old = warp_run[warp * E + e];
            warp_run[warp * E + e] = old + __popc(peers);
        }
        old = __shfl_sync(kFull, old, leader);
        my_rank[it] = old + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
    }
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += blockDim.x) {   // exclusive scan over the 8 warps
        int run = 0;
        for (int w = 0; w < 8; ++w) {
            const int c = warp_run[w * E + e];
            warp_run[w * E + e] = run;
            run += c;
        }
        block_counts[(size_t)blockIdx.x * E + e] = run;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kSortChunk / 256; ++it) {
        const int64_t s = base + it * 32 + lane;
        if (s >= N) continue;
        const int e = topk_idx[s];
        local_rank[s] = (unsigned)e < (unsigned)E ? warp_run[warp * E + e] + my_rank[it] : 0;
    }
}

// Pass 2 (one block): per expert an exclusive scan of the block counts, then offsets, padded offsets
// and the tile -> expert map.
__global__ void __launch_bounds__(1024) sort_scan_kernel(int32_t* __restrict__ block_counts, int n_blocks, int E,
                                                         int32_t* __restrict__ counts, int32_t* __restrict__ offsets,
                                                         int32_t* __restrict__ poffsets,
                                                         int32_t* __restrict__ tile_expert,
                                                         int32_t* __restrict__ n_tiles, int cap,
                                                         int32_t* __restrict__ counts_chosen) {
    grid_dependency_wait();
    grid_dependency_launch();
    __shared__ int32_t s_cnt[kMaxExperts];
    __shared__ int32_t s_poff[kMaxExperts + 1];
    __shared__ int32_t s_part[1024];
    // thread (part, e) owns a contiguous range of blocks of expert e: range sums, then the exclusive scan inside
    // the range starting from the sum of the ranges before it (two dependent passes instead of one long one)
    const int parts = E >= (int)blockDim.x ? 1 : min(16, min((int)blockDim.x / E, max(n_blocks, 1)));
    const int per = (n_blocks + parts - 1) / parts;
    for (int e0 = 0; e0 < E; e0 += blockDim.x / parts) {
        const int e = e0 + threadIdx.x % (blockDim.x / parts), part = threadIdx.x / (blockDim.x / parts);
        const bool mine = e < E && part < parts;
        const int b0 = min(n_blocks, part * per), b1 = min(n_blocks, b0 + per);
        int sum = 0;
        if (mine) {
            int b = b0;
            for (; b + 8 <= b1; b += 8) {
                int c[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) c[i] = block_counts[(size_t)(b + i) * E + e];
#pragma unroll
                for (int i = 0; i < 8; ++i) sum += c[i];
            }
            for (; b < b1; ++b) sum += block_counts[(size_t)b * E + e];
        }
        __syncthreads();                            // s_part of the previous round has been read
        if (part < parts) s_part[part * (blockDim.x / parts) + threadIdx.x % (blockDim.x / parts)] = sum;
        __syncthreads();
        if (mine) {
            int run = 0, total = 0;
            for (int q = 0; q < parts; ++q) {
                const int v = s_part[q * (blockDim.x / parts) + threadIdx.x % (blockDim.x / parts)];
                if (q < part) run += v;
                total += v;
            }
            if (part == 0) {                        // an expert keeps at most `cap` of the slots that chose it
                const int kept = min(total, cap);
                s_cnt[e] = kept;
                counts[e] = kept;
                if (counts_chosen) counts_chosen[e] = total;
            }
            int b = b0;
            for (; b + 8 <= b1; b += 8) {
                int c[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) c[i] = block_counts[(size_t)(b + i) * E + e];
#pragma unroll
                for (int i = 0; i < 8; ++i) { block_counts[(size_t)(b + i) * E + e] = run; run += c[i]; }
            }
            for (; b < b1; ++b) {
                const int c = block_counts[(size_t)b * E + e];
                block_counts[(size_t)b * E + e] = run;
                run += c;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int off = 0, poff = 0;
        for (int e = 0; e < E; ++e) {
            offsets[e] = off;
            s_poff[e] = poff;
            off += s_cnt[e];
            poff += (s_cnt[e] + kPad - 1) / kPad * kPad;
        }
        offsets[E] = off;
        s_poff[E] = poff;
        *n_tiles = poff / kPad;
    }
    __syncthreads();
    for (int e = threadIdx.x; e <= E; e += blockDim.x) poffsets[e] = s_poff[e];
    for (int e = threadIdx.x; e < E; e += blockDim.x)
        for (int tile = s_poff[e] / kPad; tile < s_poff[e + 1] / kPad; ++tile) tile_expert[tile] = e;
}

// Pass 3: final positions.  A slot whose rank among the slots of its expert is `cap` or more is dropped (-1).
__global__ void __launch_bounds__(256) sort_place_kernel(const int32_t* __restrict__ topk_idx, int64_t N, int E,
                                                         const int32_t* __restrict__ block_base,
                                                         const int32_t* __restrict__ offsets,
                                                         const int32_t* __restrict__ poffsets,
                                                         int32_t* __restrict__ prow_of_slot /* in: local rank */,
                                                         int32_t* __restrict__ row_of_slot,
                                                         int32_t* __restrict__ slot_of_row,
                                                         int32_t* __restrict__ slot_of_prow, int cap,
                                                         int* __restrict__ status) {
    grid_dependency_wait();
    grid_dependency_launch();
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const int e = topk_idx[s];
    if ((unsigned)e >= (unsigned)E) {               // second line of defence: the slot goes nowhere, the call reports it
        row_of_slot[s] = -1;
        prow_of_slot[s] = -1;
        if (status) atomicExch(status, 2);
        return;
    }
    const int within = block_base[(size_t)(s / kSortChunk) * E + e] + prow_of_slot[s];
    if (within >= cap) {
        row_of_slot[s] = -1;
        prow_of_slot[s] = -1;
        return;
    }
    const int row = offsets[e] + within;
    const int prow = poffsets[e] + within;
    row_of_slot[s] = row;
    slot_of_row[row] = (int32_t)s;
    prow_of_slot[s] = prow;
    slot_of_prow[prow] = (int32_t)s;
}

// All three passes (and the fill of slot_of_prow) in ONE block, for the few thousand slots of decode-shaped batches,
// where four launches cost more than the work.  1024 threads; chunk c holds slots [1024 c, 1024 (c + 1)), warp w of
// it the 32 slots from 1024 c + 32 w: ranks inside a warp by match_any, across the warps of a chunk by a scan over the
// per-warp counts, across chunks by the running per-expert totals - the same stable order as the three-pass sort.
__global__ void __launch_bounds__(1024) tables_small_kernel(const int32_t* __restrict__ topk_idx, int N, int E, int cap, int P,
                                                            int32_t* __restrict__ counts, int32_t* __restrict__ counts_chosen,
                                                            int32_t* __restrict__ offsets, int32_t* __restrict__ poffsets,
                                                            int32_t* __restrict__ tile_expert, int32_t* __restrict__ n_tiles,
                                                            int32_t* __restrict__ prow_of_slot, int32_t* __restrict__ row_of_slot,
                                                            int32_t* __restrict__ slot_of_row, int32_t* __restrict__ slot_of_prow,
                                                            int* __restrict__ status) {
    grid_dependency_wait();
    grid_dependency_launch();
    extern __shared__ int32_t sm[];                  // [32][E] per-warp counts of the chunk, [E] totals so far, 2 x [E+1]: 35 E + 2 ints
    int32_t* warp_run = sm;
    int32_t* total = sm + 32 * E;
    int32_t* s_off = total + E;
    int32_t* s_poff = s_off + E + 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < P; i += blockDim.x) slot_of_prow[i] = -1;
    if (cap < N)
        for (int i = threadIdx.x; i < N; i += blockDim.x) slot_of_row[i] = -1;
    for (int e = threadIdx.x; e < E; e += blockDim.x) total[e] = 0;
    const int chunks = (N + 1023) / 1024;
    int32_t rank_of[kSmallTablesMaxSlots / 1024];    // this thread's slot of every chunk: rank among its expert's slots
#pragma unroll
    for (int c = 0; c < kSmallTablesMaxSlots / 1024; ++c) {
        if (c >= chunks) break;                      // uniform
        for (int i = threadIdx.x; i < 32 * E; i += blockDim.x) warp_run[i] = 0;
        __syncthreads();
        const int s = c * 1024 + threadIdx.x;
        int e = s < N ? topk_idx[s] : -1;
        if ((unsigned)e >= (unsigned)E) e = -1;      // an id outside [0, E) counts nowhere
        const unsigned peers = __match_any_sync(kFull, e);
        if (e >= 0 && lane == __ffs(peers) - 1) warp_run[warp * E + e] = __popc(peers);
        const int in_warp = __popc(peers & ((1u << lane) - 1u));
        __syncthreads();
        for (int x = threadIdx.x; x < E; x += blockDim.x) {      // exclusive scan over the warps, on top of the earlier chunks
            int run = total[x];
            for (int w = 0; w < 32; ++w) {
                const int n = warp_run[w * E + x];
                warp_run[w * E + x] = run;
                run += n;
            }
            total[x] = run;
        }
        __syncthreads();
        rank_of[c] = e >= 0 ? warp_run[warp * E + e] + in_warp : 0;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        int off = 0, poff = 0;
        for (int e = 0; e < E; ++e) {
            const int kept = min(total[e], cap);
            s_off[e] = off;
            s_poff[e] = poff;
            off += kept;
            poff += (kept + kPad - 1) / kPad * kPad;
        }
        s_off[E] = off;
        s_poff[E] = poff;
        *n_tiles = poff / kPad;
    }
    __syncthreads();
    for (int e = threadIdx.x; e <= E; e += blockDim.x) { offsets[e] = s_off[e]; poffsets[e] = s_poff[e]; }
    for (int e = threadIdx.x; e < E; e += blockDim.x) {
        counts[e] = min(total[e], cap);
        if (counts_chosen) counts_chosen[e] = total[e];
        for (int tile = s_poff[e] / kPad; tile < s_poff[e + 1] / kPad; ++tile) tile_expert[tile] = e;
    }
#pragma unroll
    for (int c = 0; c < kSmallTablesMaxSlots / 1024; ++c) {
        if (c >= chunks) break;
        const int s = c * 1024 + threadIdx.x;
        if (s >= N) continue;
        const int e = topk_idx[s], within = rank_of[c];
        const bool bad = (unsigned)e >= (unsigned)E;
        if (bad && status) atomicExch(status, 2);
        if (bad || within >= cap) {
            row_of_slot[s] = -1;
            prow_of_slot[s] = -1;
            continue;
        }
        const int row = s_off[e] + within, prow = s_poff[e] + within;
        row_of_slot[s] = row;
        slot_of_row[row] = s;
        prow_of_slot[s] = prow;
        slot_of_prow[prow] = s;
    }
}

constexpr int kMaxParts = 8;                        // parts of a split descend contraction

// ---- Routing in two launches (k <= 8, E a multiple of 4 up to 256: every configuration of the paper) -------------
// A forward used to spend six launches between the gate logits and the experts (top-k, fill, three passes of the
// counting sort, dispatch): about 2.5 us each for work of well under a microsecond, 20 us of 128 at 3001 tokens of the
// d = 2048 widths.  Here the first kernel does the top-k and sorts inside its block, the second adds up the blocks'
// counts for itself, places the slots and moves the rows; nothing between them is a fill or a scan launch of its own.

// Where the gate logits (and the rows of x') come from: matrices in memory, or the fp32 partial results
// [parts][T][ld] of a descend launch whose contraction was cut into parts - then added in part order on the way.

// A lane's logits of its token: elements 4 (sub + 8 i) .. + 3 of the row, i < Q.  Returns bit i: element i is past E.
template <int Q>
__device__ __forceinline__ uint32_t token_logits(float* v, const float* row, int parts, int64_t part_stride, float* logits_out, int64_t t,
                                                 bool live, const float* __restrict__ b_gate, int E) {
    const int sub = threadIdx.x & 7;
    uint32_t past = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int e0 = 4 * (sub + 8 * i);
        float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (e0 < E) {
            x = *reinterpret_cast<const float4*>(row + e0);
            if (parts > 1) {                     // all parts' loads in flight together, added in part order
                float4 y[kMaxParts - 1];
#pragma unroll
                for (int s = 1; s < kMaxParts; ++s)
                    if (s < parts) y[s - 1] = *reinterpret_cast<const float4*>(row + s * part_stride + e0);
#pragma unroll
                for (int s = 1; s < kMaxParts; ++s)
                    if (s < parts) { x.x += y[s - 1].x; x.y += y[s - 1].y; x.z += y[s - 1].z; x.w += y[s - 1].w; }
            }
            if (logits_out && live) *reinterpret_cast<float4*>(logits_out + t * E + e0) = x;
            if (b_gate) { x.x += b_gate[e0]; x.y += b_gate[e0 + 1]; x.z += b_gate[e0 + 2]; x.w += b_gate[e0 + 3]; }
        } else {
            past |= 15u << (4 * i);
        }
        v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
    }
    return past;
}

// Rounds of arg-max over a token's eight lanes: a lane keeps the maxima of its Q quads in registers and the quads themselves in
// shared memory, where the winner alone strikes its element out (NaN: never a maximum, never equal) and looks its quad over
// again.  With the values in registers every lane scanned all of them in every round: issue slots bound the kernel, 34 us at
// 32768 tokens of 128 experts.
// Lane j of the eight gets the j-th choice (value, expert id).
template <int Q>
__device__ __forceinline__ void token_topk(float* v, uint32_t past, float4* quads, int k, float& my_v, int& my_e) {
    const int lane = threadIdx.x & 31, sub = lane & 7;
    my_v = -INFINITY;
    my_e = 0;
    const float none = __int_as_float(0x7fffffff);
    float most[Q];                               // maximum of each quad
#pragma unroll
    for (int i = 0; i < 4 * Q; ++i) v[i] = (past >> i) & 1u ? none : v[i] == v[i] ? v[i] : -INFINITY;     // NaN is ordered as -inf
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        most[q] = fmaxf(fmaxf(v[4 * q], v[4 * q + 1]), fmaxf(v[4 * q + 2], v[4 * q + 3]));
        quads[q * blockDim.x] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    }
    for (int j = 0; j < k; ++j) {
        float mine = most[0];
#pragma unroll
        for (int q = 1; q < Q; ++q) mine = fmaxf(mine, most[q]);
        float best = mine;
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) best = fmaxf(best, __shfl_xor_sync(kFull, best, off));
        bool wins = mine == best;
        int e = kNoExpert, at = 0, c = 0;
        float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (wins) {                              // its lowest expert id with that value: ids ascend with the quad and inside it
#pragma unroll
            for (int q = Q - 1; q >= 0; --q) at = most[q] == best ? q : at;
            x = quads[at * blockDim.x];
            c = x.x == best ? 0 : x.y == best ? 1 : x.z == best ? 2 : 3;
            e = 4 * (sub + 8 * at) + c;
        }
        const unsigned votes = __ballot_sync(kFull, wins), group = (votes >> (lane & 24)) & 0xffu;
        int from = __ffs(group) - 1;
        if (__any_sync(kFull, __popc(group) > 1)) {      // equal logits in several lanes: the lowest id of all
            int low = e;
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) low = min(low, __shfl_xor_sync(kFull, low, off));
            wins = wins && e == low;
            from = (low >> 2) & 7;
        }
        if (wins) {
            x.x = c == 0 ? none : x.x; x.y = c == 1 ? none : x.y; x.z = c == 2 ? none : x.z; x.w = c == 3 ? none : x.w;
            quads[at * blockDim.x] = x;
            const float left = fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w));
#pragma unroll
            for (int q = 0; q < Q; ++q) most[q] = at == q ? left : most[q];
        }
        const int chosen = __shfl_sync(kFull, e, (lane & 24) + from);
        if (sub == j) { my_v = best; my_e = chosen; }
    }
}

// Kernel 1: top-k with gate values as topk8_kernel, four tokens per warp, plus pass 1 of the counting sort.  Block b owns
// tokens [b TB, (b + 1) TB), TB = 4 warps iters.  Lane 8 g + j of a warp holds slot j of the warp's token g, so the lane
// order is the slot order: ranks inside a warp by match_any, across the warps by a scan over per-warp counts.
// AUX: also the block's column sums of the softmax over all E experts, for the load-balancing loss (launches of their own for
// these sums, the loss and the copies of the tables put 16 us between the logits and the experts at 2999 tokens).
constexpr int kTopkAuxWarps = 16;
template <int Q, bool AUX>   // Q float4 loads per lane: E <= 32 Q
__global__ void __launch_bounds__(AUX ? 32 * kTopkAuxWarps : 1024) topk_count_kernel(const float* __restrict__ logits, int ld, int parts, int64_t part_stride,
                                                          float* __restrict__ logits_out, const float* __restrict__ b_gate, int T,
                                                          int E, int k, int iters, int32_t* __restrict__ topk_idx,
                                                          float* __restrict__ topk_w, int32_t* __restrict__ local_rank,
                                                          int32_t* __restrict__ block_counts, int32_t* __restrict__ ex_idx,
                                                          float* __restrict__ ex_w, float* __restrict__ aux_part) {
    grid_dependency_wait();
    grid_dependency_launch();
    extern __shared__ int32_t warp_run[];            // [warps][E], then [E] the block's totals so far
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5, sub = lane & 7;
    int32_t* total = warp_run + warps * E;
    float* prob_sums = reinterpret_cast<float*>(total + E);      // AUX: [warps][E]
    float4* quads = reinterpret_cast<float4*>(prob_sums + (AUX ? warps * E : 0)) + threadIdx.x;   // [Q][threads]; E is a multiple of 4
    for (int i = threadIdx.x; i < (AUX ? 2 * warps + 1 : warps + 1) * E; i += blockDim.x) warp_run[i] = 0;   // (0 is 0.0f)
    __syncthreads();
    for (int it = 0; it < iters; ++it) {
        const int64_t t = ((int64_t)blockIdx.x * iters + it) * (4 * warps) + 4 * warp + (lane >> 3);
        const bool live = t < T;
        const float* row = logits + (live ? t : 0) * ld;
        float v[4 * Q];
        const uint32_t past = token_logits<Q>(v, row, parts, part_stride, logits_out, t, live, b_gate, E);
        if (AUX) {                                   // a token's softmax over its eight lanes, then the warp's four tokens together
            float mx = -INFINITY, sum = 0.0f, pr[4 * Q];
#pragma unroll
            for (int i = 0; i < 4 * Q; ++i)
                if (!((past >> i) & 1u)) mx = fmaxf(mx, v[i]);
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, off));
#pragma unroll
            for (int i = 0; i < 4 * Q; ++i) {
                pr[i] = !((past >> i) & 1u) && live ? expf(v[i] - mx) : 0.0f;
                sum += pr[i];
            }
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) sum += __shfl_xor_sync(kFull, sum, off);
            const float inv = live ? 1.0f / sum : 0.0f;
#pragma unroll
            for (int i = 0; i < 4 * Q; ++i) {
                float p = pr[i] * inv;
                p += __shfl_xor_sync(kFull, p, 8);
                p += __shfl_xor_sync(kFull, p, 16);
                const int e = 4 * (sub + 8 * (i >> 2)) + (i & 3);
                if (lane < 8 && e < E) prob_sums[warp * E + e] += p;
            }
        }
        float my_v;
        int my_e;
        token_topk<Q>(v, past, quads, k, my_v, my_e);
        const float top = __shfl_sync(kFull, my_v, lane & 24);
        const float ex = sub < k ? (top == -INFINITY ? 1.0f : expf(my_v - top)) : 0.0f;
        float part = ex;
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) part += __shfl_xor_sync(kFull, part, off);
        const bool slot = live && sub < k;
        const int e = slot ? my_e : -1;
        const unsigned peers = __match_any_sync(kFull, e);
        if (slot && lane == __ffs(peers) - 1) warp_run[warp * E + e] = __popc(peers);
        __syncthreads();
        for (int x = threadIdx.x; x < E; x += blockDim.x) {      // exclusive scan over the warps, on top of the earlier rounds
            int run = total[x];
            int w = 0;
            for (; w + 8 <= warps; w += 8) {
                int c[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) c[i] = warp_run[(w + i) * E + x];
#pragma unroll
                for (int i = 0; i < 8; ++i) { warp_run[(w + i) * E + x] = run; run += c[i]; }
            }
            for (; w < warps; ++w) { const int c = warp_run[w * E + x]; warp_run[w * E + x] = run; run += c; }
            total[x] = run;
        }
        __syncthreads();
        if (slot) {
            const int64_t s = t * k + sub;
            topk_idx[s] = my_e;
            topk_w[s] = ex / part;
            if (ex_idx) ex_idx[s] = my_e;
            if (ex_w) ex_w[s] = ex / part;
            local_rank[s] = warp_run[warp * E + e] + __popc(peers & ((1u << lane) - 1u));
        }
        if (it + 1 < iters) {
            __syncthreads();
            for (int i = threadIdx.x; i < warps * E; i += blockDim.x) warp_run[i] = 0;
            __syncthreads();
        }
    }
    for (int x = threadIdx.x; x < E; x += blockDim.x) {
        block_counts[(size_t)blockIdx.x * E + x] = total[x];
        if (AUX) {
            float acc = 0.0f;
            for (int w = 0; w < warps; ++w) acc += prob_sums[w * E + x];
            aux_part[(size_t)blockIdx.x * E + x] = acc;
        }
    }
}

struct PlaceArgs {
    const int32_t *topk_idx, *block_counts;
    int T, E, k, nb, tokens_per_block, splits, cap;  // nb blocks of kernel 1, each cut into `splits` blocks of this kernel
    int32_t *counts, *counts_chosen, *offsets, *poffsets, *tile_expert, *n_tiles;
    int32_t *prow_of_slot /* in: rank inside the block of kernel 1 */, *row_of_slot, *slot_of_row, *slot_of_prow;
    float* zero_word;                                // nullable: set to 0 (the loss of a layer without one)
    RouteExport ex;
    const float* aux_part;                           // nullable: [nb][E] sums of softmax probabilities
    float* aux_loss;
    float aux_coef;
    // the rows to move: [T, 16 vecs bytes] at src, or fp32 partial results [parts][T][ld] rounded to bf16
    const uint4* src;
    const float* partial;
    int parts, ld;
    int64_t part_stride;
    uint4* grouped;
    int vecs;
    bool zero_padding;                               // write zeros on the padding rows (a training step contracts over them)
    int* status;
};

constexpr int kPlaceThreads = 512, kPlaceMaxExperts = 256;
// Counts of an expert's slots before this block's, and in all; rows before the expert, unpadded and padded.
struct PlaceShared { int32_t base[kPlaceMaxExperts], total[kPlaceMaxExperts], off[kPlaceMaxExperts + 1], poff[kPlaceMaxExperts + 1]; };

// The placement from the counts on: tokens [first, last) of this block, slot_of(t, e, rank) giving lane j < k of a warp its slot's
// expert and rank behind sh.base (MOVE 0: slot_of(s, e, rank) those of slot s); then this block's share of everything else.
template <int MOVE, typename Slot>
__device__ __forceinline__ void place_from_counts(const PlaceArgs& p, PlaceShared& sh, int64_t first, int64_t last, Slot slot_of) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, E = p.E, nparts = min(16, kPlaceThreads / E);
    constexpr int kWarps = kPlaceThreads / 32;
    int32_t *s_base = sh.base, *s_total = sh.total, *s_off = sh.off, *s_poff = sh.poff;
    __syncthreads();
    if (warp == 0) {                                 // offsets: lane l scans the experts [l per, (l + 1) per)
        const int per = (E + 31) / 32, e0 = min(E, lane * per), e1 = min(E, e0 + per);
        int rows = 0, padded = 0;
        for (int e = e0; e < e1; ++e) {
            const int kept = min(s_total[e], p.cap);
            rows += kept;
            padded += (kept + kPad - 1) / kPad * kPad;
        }
        int r = rows, q = padded;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(kFull, r, o), c = __shfl_up_sync(kFull, q, o);
            if (lane >= o) { r += a; q += c; }
        }
        int off = r - rows, poff = q - padded;
        for (int e = e0; e < e1; ++e) {
            const int kept = min(s_total[e], p.cap);
            s_off[e] = off;
            s_poff[e] = poff;
            off += kept;
            poff += (kept + kPad - 1) / kPad * kPad;
        }
        if (lane == 31) { s_off[E] = off; s_poff[E] = poff; }
    }
    __syncthreads();
    // ---- this block's tokens
    auto place = [&](int64_t s, int e, int rank) {   // one slot's tables; its padded row or -1
        int row = -1, prow = -1;
        if ((unsigned)e >= (unsigned)E) {            // second line of defence: the slot goes nowhere, the call reports it
            if (p.status) atomicExch(p.status, 2);
        } else {
            const int within = s_base[e] + rank;
            if (within < p.cap) {                    // else dropped under a capacity limit
                row = s_off[e] + within;
                prow = s_poff[e] + within;
                p.slot_of_row[row] = (int32_t)s;
                p.slot_of_prow[prow] = (int32_t)s;
            }
        }
        p.row_of_slot[s] = row;
        p.prow_of_slot[s] = prow;
        if (p.ex.row_of_slot) p.ex.row_of_slot[s] = row;
        if (p.ex.slot_of_row && row >= 0) p.ex.slot_of_row[row] = (int32_t)s;
        return prow;
    };
    // No rows to move: a thread a slot.  (A warp a token, eight of its lanes at work on three or four tokens one after another:
    // the routing call of 16384 tokens 35.2 us, so 33.2.)
    if (MOVE == 0) {
        for (int64_t s = first * p.k + tid; s < last * p.k; s += kPlaceThreads) {
            int e, rank;
            slot_of(s, e, rank);
            place(s, e, rank);
        }
    } else
    for (int64_t t = first + warp; t < last; t += kWarps) {
        uint4 v0 = make_uint4(0, 0, 0, 0), v1 = v0;
        if (MOVE == 1) {                             // the first 64 pieces of the row are on their way before its place is known
            if (lane < p.vecs) v0 = __ldg(p.src + t * p.vecs + lane);
            if (lane + 32 < p.vecs) v1 = __ldg(p.src + t * p.vecs + lane + 32);
        }
        int prow = -1;
        if (lane < p.k) {
            int e, rank;
            slot_of(t, e, rank);
            prow = place(t * p.k + lane, e, rank);
        }
        for (int c = lane; c - lane < p.vecs; c += 64) {
            if (MOVE == 1) {
                if (c >= 64) {
                    if (c < p.vecs) v0 = __ldg(p.src + t * p.vecs + c);
                    if (c + 32 < p.vecs) v1 = __ldg(p.src + t * p.vecs + c + 32);
                }
            } else {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int cc = c + 32 * h;
                    if (cc >= p.vecs) continue;
                    const float* from = p.partial + t * p.ld + 8 * cc;
                    float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f), d = a, x[kMaxParts], y[kMaxParts];
#pragma unroll
                    for (int s = 0; s < kMaxParts; ++s)
                        if (s < p.parts) {
                            x[s] = *reinterpret_cast<const float4*>(from + s * p.part_stride);
                            y[s] = *reinterpret_cast<const float4*>(from + s * p.part_stride + 4);
                        }
#pragma unroll
                    for (int s = 0; s < kMaxParts; ++s)
                        if (s < p.parts) {
                            a.x += x[s].x; a.y += x[s].y; a.z += x[s].z; a.w += x[s].w;
                            d.x += y[s].x; d.y += y[s].y; d.z += y[s].z; d.w += y[s].w;
                        }
                    __nv_bfloat162 o[4] = {__floats2bfloat162_rn(a.x, a.y), __floats2bfloat162_rn(a.z, a.w),
                                           __floats2bfloat162_rn(d.x, d.y), __floats2bfloat162_rn(d.z, d.w)};
                    (h ? v1 : v0) = *reinterpret_cast<uint4*>(o);
                }
            }
            for (int j = 0; j < p.k; ++j) {
                const int to = __shfl_sync(kFull, prow, j);
                if (to < 0) continue;                // uniform
                if (c < p.vecs) p.grouped[(int64_t)to * p.vecs + c] = v0;
                if (c + 32 < p.vecs) p.grouped[(int64_t)to * p.vecs + c + 32] = v1;
            }
        }
    }
    // ---- padding rows: the gaps behind the experts' rows, dealt out over all blocks
    const int share = max(1, (int)gridDim.x / E);    // blocks per expert
    for (int e = blockIdx.x / share; e < E; e += gridDim.x / share) {
        const int r0 = s_poff[e] + (s_off[e + 1] - s_off[e]), r1 = s_poff[e + 1];
        if (MOVE == 0 || p.zero_padding)             // (nothing after the dispatch of an inference forward looks at a padding row)
            for (int r = r0 + (int)(blockIdx.x % share) * kPlaceThreads + tid; r < r1; r += share * kPlaceThreads) p.slot_of_prow[r] = -1;
        if (MOVE != 0 && p.zero_padding)
            for (int r = r0 + (int)(blockIdx.x % share) * kWarps + warp; r < r1; r += share * kWarps)
                for (int c = lane; c < p.vecs; c += 32) p.grouped[(int64_t)r * p.vecs + c] = make_uint4(0, 0, 0, 0);
        if (blockIdx.x % share == 0)
            for (int tile = s_poff[e] / kPad + tid; tile < s_poff[e + 1] / kPad; tile += kPlaceThreads) p.tile_expert[tile] = e;
    }
    if (p.cap < kNoCapacity)                         // rows past the kept ones exist only under a capacity limit
        for (int64_t r = s_off[E] + (int64_t)blockIdx.x * kPlaceThreads + tid; r < (int64_t)p.T * p.k; r += (int64_t)gridDim.x * kPlaceThreads)
        {
            p.slot_of_row[r] = -1;
            if (p.ex.slot_of_row) p.ex.slot_of_row[r] = -1;
        }
    if (p.aux_part && blockIdx.x == gridDim.x - 1) { // the loss, coef E sum_e f_e P_e, on the block with the fewest tokens
        __shared__ float s_term[kPlaceMaxExperts];
        __shared__ float sums[kPlaceThreads];
        const int e = tid % E, part = tid / E;
        float acc = 0.0f;
        if (part < nparts) {
#pragma unroll 8
            for (int row = part; row < p.nb; row += nparts) acc += p.aux_part[(size_t)row * E + e];
        }
        sums[tid] = acc;
        __syncthreads();
        if (tid < E) {
            float P = 0.0f;
            for (int q = 0; q < nparts; ++q) P += sums[q * E + tid];
            s_term[tid] = ((float)s_total[tid] / ((float)p.T * (float)p.k)) * (P / (float)p.T);
        }
        __syncthreads();
        if (warp == 0) {
            float v = 0.0f;
            for (int x = lane; x < E; x += 32) v += s_term[x];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
            if (lane == 0) {
                const float loss = p.aux_coef * (float)E * v;
                *p.aux_loss = loss;
                if (p.ex.aux_loss) *p.ex.aux_loss = loss;
            }
        }
    }
    if (blockIdx.x == 0) {
        for (int e = tid; e <= E; e += kPlaceThreads) {
            p.offsets[e] = s_off[e];
            p.poffsets[e] = s_poff[e];
            if (p.ex.offsets) p.ex.offsets[e] = s_off[e];
        }
        for (int e = tid; e < E; e += kPlaceThreads) {
            p.counts[e] = min(s_total[e], p.cap);
            if (p.counts_chosen) p.counts_chosen[e] = s_total[e];
            if (p.ex.counts) p.ex.counts[e] = min(s_total[e], p.cap);
            if (p.ex.counts_chosen) p.ex.counts_chosen[e] = s_total[e];
        }
        if (tid == 0) {
            *p.n_tiles = s_poff[E] / kPad;
            if (p.zero_word) *p.zero_word = 0.0f;
        }
    }
}


// Kernel 2: the whole placement, and the dispatch as a scatter: a warp reads the row of a token once and writes it to
// its k grouped rows (the gather form reads it k times).  Every block adds up the counts of all blocks of kernel 1 for
// itself (a few tens of KB from L2), which takes less than a launch of a scan kernel.
// MOVE 0: tables only; 1: rows of a matrix; 2: rows from partial results.
template <int MOVE>
__global__ void __launch_bounds__(kPlaceThreads) place_kernel(const PlaceArgs p) {
    grid_dependency_wait();
    grid_dependency_launch();
    __shared__ int32_t s_all[kPlaceThreads], s_below[kPlaceThreads];        // [parts][E]
    __shared__ PlaceShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kWarps = kPlaceThreads / 32;
    const int E = p.E, nparts = min(16, kPlaceThreads / E);
    const int b = blockIdx.x / p.splits;             // the block of kernel 1 whose slots these are
    const int per_split = (p.tokens_per_block + p.splits - 1) / p.splits;
    const int64_t first = (int64_t)b * p.tokens_per_block + (int64_t)(blockIdx.x - b * p.splits) * per_split;
    const int64_t last = min(min(first + per_split, (int64_t)(b + 1) * p.tokens_per_block), (int64_t)p.T);
    // the warp's first token (the thread's first slot): experts and ranks are on their way while the counts are added up
    int next_e = 0, next_rank = 0;
    const int64_t s_first = MOVE == 0 ? first * p.k + tid : (first + warp) * p.k + lane;
    if (MOVE == 0 ? s_first < last * p.k : first + warp < last && lane < p.k) {
        next_e = p.topk_idx[s_first];
        next_rank = p.prow_of_slot[s_first];
    }
    {
        const int e = tid % E, part = tid / E;       // neighbouring threads on neighbouring experts
        int all = 0, below = 0;
        if (part < nparts) {
            for (int row = part; row < p.nb; row += 16 * nparts) {
                int c[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) c[i] = row + i * nparts < p.nb ? p.block_counts[(size_t)(row + i * nparts) * E + e] : 0;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    all += c[i];
                    if (row + i * nparts < b) below += c[i];
                }
            }
        }
        s_all[tid] = all;
        s_below[tid] = below;
    }
    __syncthreads();
    if (tid < E) {
        int all = 0, below = 0;
        for (int q = 0; q < nparts; ++q) {
            all += s_all[q * E + tid];
            below += s_below[q * E + tid];
        }
        sh.total[tid] = all;
        sh.base[tid] = below;
    }
    place_from_counts<MOVE>(p, sh, first, last, [&](int64_t t, int& e, int& rank) {
        const int64_t s = MOVE == 0 ? t + kPlaceThreads : (t + kWarps) * p.k + lane;       // the next one
        e = next_e;
        rank = next_rank;
        if (MOVE == 0 ? s < last * p.k : t + kWarps < last) { next_e = p.topk_idx[s]; next_rank = p.prow_of_slot[s]; }
    });
}

// Both in one launch, for up to kOneLaunchTokens tokens: a cluster of eight blocks does the top-k of all tokens, an eighth in each
// block, and the blocks hand each other their counts through distributed shared memory; every cluster does the same and then
// places and moves its own share of its blocks' tokens.  The repetition costs some L2 reads; the hand-over through memory
// (a launch's end, the next one's start, the counts and slots read back) cost about 3 us of a forward of 45 to 54.
constexpr int kOneLaunchTokens = 512, kRouteCluster = 8;
struct RouteArgs {
    const float* logits;
    int ld, parts;
    int64_t part_stride;
    const float* b_gate;
    int32_t* topk_idx;
    float* topk_w;
    int per_block;                                   // tokens of a block, at most four for each of its warps
};
// MOVE as above.
template <int Q, int MOVE>
__global__ void __cluster_dims__(kRouteCluster, 1, 1) __launch_bounds__(kPlaceThreads) route_cluster_kernel(const RouteArgs r, const PlaceArgs p) {
    constexpr int kWarps = kPlaceThreads / 32;
    extern __shared__ float4 route_quads[];          // [Q][threads]; then the counts of the warps
    int32_t* warp_run = reinterpret_cast<int32_t*>(route_quads + Q * kPlaceThreads);      // [kWarps][E]
    __shared__ PlaceShared sh;
    __shared__ int32_t counts[kRouteCluster][kPlaceMaxExperts];
    __shared__ int16_t s_expert[kOneLaunchTokens], s_rank[kOneLaunchTokens];   // slots of this block: 64 tokens of up to eight
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, sub = lane & 7, E = p.E;
    const int rank_in = blockIdx.x % kRouteCluster, cluster = blockIdx.x / kRouteCluster, clusters = gridDim.x / kRouteCluster;
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");       // (that all blocks of the cluster have started)
    for (int i = tid; i < kWarps * E; i += kPlaceThreads) warp_run[i] = 0;
    grid_dependency_wait();
    grid_dependency_launch();
    const int first = rank_in * r.per_block, here = 4 * warp + (lane >> 3), t = first + here;
    const bool live = here < r.per_block && t < p.T;
    float v[4 * Q], my_v;
    int my_e;
    const uint32_t past = token_logits<Q>(v, r.logits + (int64_t)(live ? t : 0) * r.ld, r.parts, r.part_stride, nullptr, t, live, r.b_gate, E);
    token_topk<Q>(v, past, route_quads + tid, p.k, my_v, my_e);
    const float top = __shfl_sync(kFull, my_v, lane & 24);
    const float ex = sub < p.k ? (top == -INFINITY ? 1.0f : expf(my_v - top)) : 0.0f;
    float part = ex;
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) part += __shfl_xor_sync(kFull, part, off);
    const bool slot = live && sub < p.k;
    const int e = slot ? my_e : -1;
    const unsigned peers = __match_any_sync(kFull, e);
    __syncthreads();
    if (slot && lane == __ffs(peers) - 1) warp_run[warp * E + e] = __popc(peers);
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (tid < E) {                                   // over the warps, then to all blocks of the cluster
        int run = 0, c[kWarps];
#pragma unroll
        for (int w = 0; w < kWarps; ++w) c[w] = warp_run[w * E + tid];
#pragma unroll
        for (int w = 0; w < kWarps; ++w) { warp_run[w * E + tid] = run; run += c[w]; }
        const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&counts[rank_in][tid]);
#pragma unroll
        for (int q = 0; q < kRouteCluster; ++q)
            asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %0, %1;\n\tst.shared::cluster.b32 [a], %2;\n\t}" ::"r"(mine), "r"(q), "r"(run) : "memory");
    }
    __syncthreads();
    if (slot) {
        s_expert[here * p.k + sub] = (int16_t)e;
        s_rank[here * p.k + sub] = (int16_t)(warp_run[warp * E + e] + __popc(peers & ((1u << lane) - 1u)));
        if (cluster == 0) {
            const int s = t * p.k + sub;
            r.topk_idx[s] = my_e;
            r.topk_w[s] = ex / part;
            if (p.ex.topk_idx) p.ex.topk_idx[s] = my_e;
            if (p.ex.topk_w) p.ex.topk_w[s] = ex / part;
        }
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");   // all counts are here
    if (tid < E) {
        int all = 0, below = 0;
#pragma unroll
        for (int q = 0; q < kRouteCluster; ++q) {
            const int c = counts[q][tid];
            all += c;
            if (q < rank_in) below += c;
        }
        sh.total[tid] = all;
        sh.base[tid] = below;
    }
    const int share = (r.per_block + clusters - 1) / clusters, from = min(first + cluster * share, first + r.per_block);
    const int to = min(min(from + share, first + r.per_block), p.T);
    place_from_counts<MOVE>(p, sh, from, to, [&](int64_t tok, int& ex_id, int& rank) {
        const int at = MOVE == 0 ? (int)tok - first * p.k : ((int)tok - first) * p.k + lane;     // MOVE 0: tok is the slot
        ex_id = s_expert[at];
        rank = s_rank[at];
    });
}

}  // namespace

cudaError_t launch_topk(const float* logits, const float* b_gate, int T, int E, int k, int32_t* topk_idx,
                        float* topk_w, cudaStream_t stream) {
    if (T == 0) return cudaSuccess;
    const int warps = 8;
    dim3 grid((T + warps - 1) / warps), block(warps * 32);
    const int vpl = (E + 31) / 32;
#define BIGMAC_TOPK(V)                                                                                   \
    do {                                                                                                 \
        if (k <= 32) return launch_chained(topk_kernel<V, true>, grid, block, 0, stream, logits, b_gate, T, E, k, topk_idx, topk_w);  \
        else return launch_chained(topk_kernel<V, false>, grid, block, 0, stream, logits, b_gate, T, E, k, topk_idx, topk_w);          \
    } while (0)
    if (vpl <= 1) BIGMAC_TOPK(1);
    else if (vpl <= 2) BIGMAC_TOPK(2);
    else if (vpl <= 4) BIGMAC_TOPK(4);
    else if (vpl <= 8) BIGMAC_TOPK(8);
    else if (vpl <= 16) BIGMAC_TOPK(16);
    else BIGMAC_TOPK(32);
#undef BIGMAC_TOPK
    return cudaGetLastError();
}

cudaError_t launch_tables(const Tables& tb, int T, int E, int k, int cap, cudaStream_t stream, int* status) {
    const int64_t N = (int64_t)T * k;
    const int64_t P = padded_rows_max(N, E);
    if (tables_kernel_count(N, E) == 1) {
        return launch_chained(tables_small_kernel, 1, 1024, sizeof(int32_t) * (35 * E + 2), stream, tb.topk_idx, (int)N, E, cap,
                              (int)P, tb.counts, tb.counts_chosen, tb.offsets, tb.poffsets, tb.tile_expert, tb.n_tiles,
                              tb.prow_of_slot, tb.row_of_slot, tb.slot_of_row, tb.slot_of_prow, status);
    }
    cudaError_t err = cudaMemsetAsync(tb.slot_of_prow, 0xff, sizeof(int32_t) * P, stream);
    if (err != cudaSuccess) return err;
    if (cap < N) {                                   // rows past the kept ones exist only under a capacity limit
        err = cudaMemsetAsync(tb.slot_of_row, 0xff, sizeof(int32_t) * N, stream);
        if (err != cudaSuccess) return err;
    }
    const int nb = sort_blocks(N);
    if (nb > 0) {
        err = launch_chained(sort_local_kernel, nb, 256, sizeof(int32_t) * 8 * E, stream, tb.topk_idx, N, E, tb.prow_of_slot,
                             tb.block_counts);
        if (err != cudaSuccess) return err;
    }
    err = launch_chained(sort_scan_kernel, 1, 1024, 0, stream, tb.block_counts, nb, E, tb.counts, tb.offsets, tb.poffsets,
                         tb.tile_expert, tb.n_tiles, cap, tb.counts_chosen);
    if (err != cudaSuccess) return err;
    if (N > 0)
        err = launch_chained(sort_place_kernel, (unsigned)((N + 255) / 256), 256, 0, stream, tb.topk_idx, N, E, tb.block_counts,
                             tb.offsets, tb.poffsets, tb.prow_of_slot, tb.row_of_slot, tb.slot_of_row, tb.slot_of_prow, cap,
                             status);
    return err;
}

// The two-launch form wants a lane per slot of a token, eight lanes per token, and at most 32 logits per lane.
bool route_fused_supported(int E, int k) { return k <= 8 && E % 4 == 0 && E <= kPlaceMaxExperts; }

bool route_one_launch(const RouteSource& src, const RouteMove& mv, int T, int E) {
    return T <= kOneLaunchTokens && E <= 128 && !src.aux_part && !src.logits_out;
}

cudaError_t launch_route_fused(const RouteSource& src, const RouteMove& mv, const RouteExport& ex, const float* b_gate, const Tables& tb,
                               int T, int E, int k, int cap, float* zero_word, int sm_count, cudaStream_t stream, int* status,
                               int which) {
    // As many blocks as there are SMs (and rows in block_counts) at most, 32 tokens in each at least: top-k is bound by
    // issue and latency inside a block, so few fat blocks are slow (128 tokens a block: 2 us more at 512 tokens), and the
    // second kernel reads all blocks' counts, so more blocks than SMs buy nothing.
    const int nb_max = tb.block_rows < sm_count ? tb.block_rows : sm_count;
    int per = (T + nb_max - 1) / nb_max;
    if (per < 32) per = 32;
    const int most = src.aux_part ? kTopkAuxWarps : 32, warps = per < 4 * most ? (per + 3) / 4 : most, iters = (per + 4 * warps - 1) / (4 * warps);
    per = 4 * warps * iters;
    const int nb = (T + per - 1) / per;
    if (which == 0) {                                // (which 2 has no first launch)
        const int quads = E <= 32 ? 1 : E <= 64 ? 2 : E <= 128 ? 4 : 8;          // 160 KB at most
        const size_t smem = sizeof(int32_t) * (size_t)(src.aux_part ? 2 * warps + 1 : warps + 1) * E + (size_t)quads * warps * 32 * sizeof(float4);
#define BIGMAC_TOPK_COUNT(Q)                                                                                                       \
    do {                                                                                                                           \
        const auto kernel = src.aux_part ? topk_count_kernel<Q, true> : topk_count_kernel<Q, false>;                              \
        static PerDeviceOnce once;                                                                                                 \
        int dev;                                                                                                                   \
        if (once.needed(&dev)) {                                                                                                   \
            cudaError_t e = cudaFuncSetAttribute(topk_count_kernel<Q, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 163840); \
            if (e == cudaSuccess) e = cudaFuncSetAttribute(topk_count_kernel<Q, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 172032); \
            if (e != cudaSuccess) return e;                                                                                        \
            once.mark(dev);                                                                                                        \
        }                                                                                                                          \
        return launch_chained(kernel, nb, warps * 32, smem, stream, src.logits, src.ld, src.parts, src.part_stride,               \
                              src.logits_out, b_gate, T, E, k, iters, tb.topk_idx, tb.topk_w, tb.prow_of_slot, tb.block_counts,    \
                              ex.topk_idx, ex.topk_w, src.aux_part);                                                               \
    } while (0)
        if (E <= 32) BIGMAC_TOPK_COUNT(1);
        if (E <= 64) BIGMAC_TOPK_COUNT(2);
        if (E <= 128) BIGMAC_TOPK_COUNT(4);
        BIGMAC_TOPK_COUNT(8);
#undef BIGMAC_TOPK_COUNT
    }
    PlaceArgs p{};
    p.topk_idx = tb.topk_idx; p.block_counts = tb.block_counts;
    p.T = T; p.E = E; p.k = k; p.nb = nb; p.tokens_per_block = per; p.cap = cap;
    p.splits = 2 * sm_count / nb;                   // about two blocks per SM, four tokens in each at least
    if (p.splits > per / 4) p.splits = per / 4;
    if (p.splits < 1) p.splits = 1;
    p.counts = tb.counts; p.counts_chosen = tb.counts_chosen; p.offsets = tb.offsets; p.poffsets = tb.poffsets;
    p.tile_expert = tb.tile_expert; p.n_tiles = tb.n_tiles; p.prow_of_slot = tb.prow_of_slot; p.row_of_slot = tb.row_of_slot;
    p.slot_of_row = tb.slot_of_row; p.slot_of_prow = tb.slot_of_prow; p.zero_word = zero_word; p.status = status;
    p.ex = ex; p.aux_part = src.aux_part; p.aux_loss = src.aux_loss; p.aux_coef = src.aux_coef;
    p.src = (const uint4*)mv.src; p.partial = mv.partial; p.parts = mv.parts; p.ld = mv.ld; p.part_stride = mv.part_stride;
    p.grouped = (uint4*)mv.grouped; p.vecs = mv.row_bytes / 16; p.zero_padding = mv.zero_padding;
    if (which == 2) {
        RouteArgs r{src.logits, src.ld, src.parts, src.part_stride, b_gate, tb.topk_idx, tb.topk_w, (T + kRouteCluster - 1) / kRouteCluster};
        // about four tokens a block to move, up to twelve clusters (sixteen do not fit the chip at once: 512 tokens 55 -> 61 us)
        int clusters = (r.per_block + 3) / 4;
        if (clusters > 12) clusters = 12;
        const int quads = E <= 32 ? 1 : E <= 64 ? 2 : 4;
        const size_t smem = (size_t)quads * kPlaceThreads * sizeof(float4) + sizeof(int32_t) * (kPlaceThreads / 32) * E;     // 40 KB at most
#define BIGMAC_ROUTE(Q)                                                                                                            \
    do {                                                                                                                           \
        const auto kernel = !mv.grouped ? route_cluster_kernel<Q, 0> : mv.partial ? route_cluster_kernel<Q, 2> : route_cluster_kernel<Q, 1>; \
        static PerDeviceOnce once;                                                                                                 \
        int dev;                                                                                                                   \
        if (once.needed(&dev)) {                                                                                                   \
            cudaError_t e = cudaFuncSetAttribute(route_cluster_kernel<Q, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 49152);  \
            if (e == cudaSuccess) e = cudaFuncSetAttribute(route_cluster_kernel<Q, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 49152); \
            if (e == cudaSuccess) e = cudaFuncSetAttribute(route_cluster_kernel<Q, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, 49152); \
            if (e != cudaSuccess) return e;                                                                                        \
            once.mark(dev);                                                                                                        \
        }                                                                                                                          \
        return launch_chained(kernel, kRouteCluster * clusters, kPlaceThreads, smem, stream, r, p);                                \
    } while (0)
        if (E <= 32) BIGMAC_ROUTE(1);
        if (E <= 64) BIGMAC_ROUTE(2);
        BIGMAC_ROUTE(4);
#undef BIGMAC_ROUTE
    }
    if (!mv.grouped) return launch_chained(place_kernel<0>, nb * p.splits, kPlaceThreads, 0, stream, p);
    if (!mv.partial) return launch_chained(place_kernel<1>, nb * p.splits, kPlaceThreads, 0, stream, p);
    return launch_chained(place_kernel<2>, nb * p.splits, kPlaceThreads, 0, stream, p);
}

}  // namespace bigmac
