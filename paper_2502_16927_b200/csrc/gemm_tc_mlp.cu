// Inference forward of the experts in one kernel: u = W2_e sigma(W1_e x') for the rows of every expert's segment (Eq. 4),
// the hidden activations never leaving the SM.
//
// The weights are the A operand: 128 rows of W1_e (hidden units) or of W2_e (columns of u) are the M of an MMA and the
// tokens of a row tile its N, so an expert with 8 rows costs MMAs of N = 16 and not a 128-row tile of padding, and all
// weight traffic is one stream of 16 KB boxes through one ring.  A work item is (row tile of up to NT tokens, slice of the
// hidden width); it walks its slice in chunks of 128 hidden units:
//   GEMM1   acc1[c % 2] (128 hidden x n tokens, tensor memory) = W1_e[chunk, :] X^T        r / 64 boxes
//   sigma   16 epilogue warps read acc1, apply the activation and write it as bf16 to shared memory in the MN-major layout
//           of a B operand (a[c % 2], 128 hidden x n): lane = hidden unit = contraction row, so a lane's values are adjacent
//   GEMM2   acc2 (r x n, tensor memory, r / 128 tiles) += W2_e[:, chunk] a[c % 2]          2 r / 128 boxes
// GEMM1 runs one chunk ahead of GEMM2.  After the last chunk acc2 leaves as rows of `out`, by slot: bf16 [slots][r], or fp32 [slices][slots][r].  The
// combine kernel adds a token's k slots and the slices in order, so slices need no other exchange, and padding rows are never
// written.  (An issuing thread, a producer thread and a ring for either GEMM, so that their MMAs overlap: 1.9 -> 1.65 us for a
// chunk of 128 tokens, which is what shared memory delivers operands, weights and activations at, but longer until the
// first activation; 64 tokens 45.7 -> 47.2 us a forward, 512 53.9 -> 56.1, 3001 the same.)
// The experts' row offsets are brought to shared memory in one round trip and looked up there: from the number of tiles to a
// tile's expert to its rows, three dependent loads stood before the first box.
//
// What bounds it: few tokens, the stream of weights (67 MB at 64 experts of 2 x 256 x 1024); many tokens, the MMAs
// (M = 128, N = 128: shared memory delivers both operands at just the rate of the tensor pipe) and the activation.
// Ring of 16 KB stages: NT = 128: 6 (96 KB in flight per SM; about 44 KB cover the DRAM latency at the full rate), beside X
// 64 KB and two activation buffers of 32 KB at r = 256; NT = 64: 8, for r up to 512 (X 64 KB, activations 2 x 16 KB).
#include "tc_common.cuh"

namespace bigmac {

using namespace tc;

namespace {

constexpr int HC = 128;                                  // hidden units per chunk
constexpr uint32_t BOX_BYTES = 128 * BK * 2;             // one ring stage: 128 weight rows x 64 contraction elements
constexpr int kMlpEpiWarps = 16;
constexpr int kMlpThreads = (2 + kMlpEpiWarps) * 32;

struct MlpParams {
    void* out;               // [slices][slots][r] fp32, or [slots][r] bf16 if there is one slice
    int64_t slots;
    int r, h, act, E;
    MlpSlicing sl;
    const int32_t *poffsets, *counts, *slot_of_prow;
    int max_tiles;
    int* status;
};

// A work item as every role sees it; n = 0: nothing to do (the second half of a short tile).
struct MlpItem {
    int expert, row0, rows, n, c0, chunks, slice;
};

// s_off: padded row offsets of the experts, s_pad: padding rows behind each (both in shared memory)
template <int NT>
__device__ __forceinline__ MlpItem mlp_item(const MlpParams& p, int tiles, int slices, const int32_t* s_off, const uint8_t* s_pad, int i) {
    // all first halves of the tiles come before the second ones (NT = 64), most of which are empty where experts are short
    MlpItem t;
    const int half = NT < 128 && i >= tiles * slices ? 1 : 0, j = i - half * tiles * slices, tile = j >> (__ffs(slices) - 1);
    t.slice = j - tile * slices;
    t.row0 = tile * kPad + half * NT;
    int lo = 0, hi = p.E;                                // largest expert whose rows begin at or before the tile
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (s_off[mid] <= tile * kPad) lo = mid; else hi = mid;
    }
    t.expert = lo;
    t.rows = min(NT, s_off[lo + 1] - (int)s_pad[lo] - t.row0);
    t.n = t.rows > 0 ? (t.rows + 15) / 16 * 16 : 0;
    t.c0 = t.slice * p.sl.chunks >> (__ffs(slices) - 1);
    t.chunks = ((t.slice + 1) * p.sl.chunks >> (__ffs(slices) - 1)) - t.c0;
    return t;
}

template <int NT, int STAGES>
__global__ void __launch_bounds__(kMlpThreads, 1)
fused_mlp_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w1,
                 const __grid_constant__ CUtensorMap map_w2, const MlpParams p) {
    constexpr uint32_t A_CHUNKS = NT / 64;               // 64-token column blocks of an activation buffer
    constexpr uint32_t ACT_BYTES = A_CHUNKS * HC * 128;
    constexpr uint32_t XKB_BYTES = NT * BK * 2;          // one 64-deep k slice of X
    const int KB1 = p.r / BK, MT = (p.r + 127) / 128;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* s_ring = smem;
    uint8_t* s_act = s_ring + STAGES * BOX_BYTES;        // [2]
    uint8_t* s_x = s_act + 2 * ACT_BYTES;
    uint64_t* bars = (uint64_t*)(s_x + (uint32_t)KB1 * XKB_BYTES);
    uint64_t* full = bars;              uint64_t* empty = bars + STAGES;
    uint64_t* x_full = bars + 2 * STAGES;
    uint64_t* x_empty = x_full + 1;
    uint64_t* acc1_full = x_full + 2;   uint64_t* acc1_empty = x_full + 4;       // [2] each
    uint64_t* act_full = x_full + 6;    uint64_t* act_empty = x_full + 8;        // [2] each
    uint64_t* acc2_full = x_full + 10;  uint64_t* acc2_empty = x_full + 11;
    uint32_t* tmem_slot = (uint32_t*)(x_full + 12);
    volatile int* dead = (volatile int*)(tmem_slot + 1);
    int32_t* s_off = (int32_t*)(tmem_slot + 4);          // [E + 1]
    uint8_t* s_pad = (uint8_t*)(s_off + p.E + 1);        // [E]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 32) {                             // the maps are on their way while the barriers are set up
        prefetch_tensormap(&map_x);
        prefetch_tensormap(&map_w1);
        prefetch_tensormap(&map_w2);
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(x_full, 1); mbar_init(x_empty, 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(&acc1_full[s], 1); mbar_init(&acc1_empty[s], kMlpEpiWarps);
            mbar_init(&act_full[s], kMlpEpiWarps); mbar_init(&act_empty[s], 1);
        }
        mbar_init(acc2_full, 1); mbar_init(acc2_empty, kMlpEpiWarps);
        *dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // Chained launch: everything above touched no global memory and may have run while the kernel before this one in
    // the stream was still working.  Tensor memory is held, so the next kernel of the stream may be set up in turn;
    // from the wait on, the predecessor's results are complete.
    grid_dependency_launch();
    grid_dependency_wait();
    for (int e = threadIdx.x; e <= p.E; e += kMlpThreads) {
        s_off[e] = p.poffsets[e];
        if (e < p.E) s_pad[e] = (uint8_t)((kPad - p.counts[e] % kPad) % kPad);
    }
    __syncthreads();
    const uint32_t tmem_base = *tmem_slot, acc2_tmem = tmem_base + 2 * NT;
    const int tiles = min(s_off[p.E] / kPad, p.max_tiles), slices = mlp_slices(p.sl, tiles), total = tiles * (128 / NT) * slices;

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer: X once per item, then the weight boxes
        if (elect_one()) {
            uint32_t s = 0, phase = 1, local = 0;
            auto box = [&](const CUtensorMap* map, int c0, int c1) {
                mbar_wait_lean(&empty[s], phase, dead, p.status);
                mbar_expect_tx(&full[s], BOX_BYTES);
                tma_load_2d(s_ring + s * BOX_BYTES, map, &full[s], c0, c1);
                if (++s == STAGES) { s = 0; phase ^= 1; }
            };
            for (int i = blockIdx.x; i < total; i += gridDim.x) {
                const MlpItem t = mlp_item<NT>(p, tiles, slices, s_off, s_pad, i);
                if (t.n == 0) continue;
                mbar_wait_lean(x_empty, (local & 1) ^ 1, dead, p.status);
                ++local;
                mbar_expect_tx(x_full, (uint32_t)(KB1 * t.n) * BK * 2);
                for (int kb = 0; kb < KB1; ++kb)
                    for (int j = 0; j < t.n; j += 16) tma_load_2d(s_x + kb * XKB_BYTES + j * 128, &map_x, x_full, kb * BK, t.row0 + j);
                const int w1_row = t.expert * p.h + t.c0 * HC, w2_row = t.expert * p.r;
                for (int c = 0; c <= t.chunks; ++c) {    // in the order of the MMAs: W1 of chunk c, W2 of chunk c - 1
                    if (c < t.chunks)
                        for (int kb = 0; kb < KB1; ++kb) box(&map_w1, kb * BK, w1_row + c * HC);
                    if (c > 0)
                        for (int m = 0; m < MT; ++m)
                            for (int kh = 0; kh < 2; ++kh) box(&map_w2, (t.c0 + c - 1) * HC + kh * BK, w2_row + m * 128);
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (one thread)
        if (elect_one()) {
            const uint64_t d_ring = smem_desc(smem_u32(s_ring), 16, 1024), d_x = smem_desc(smem_u32(s_x), 16, 1024);
            const uint64_t d_act = smem_desc(smem_u32(s_act), HC * 128, 1024);   // MN-major, 64-token blocks HC rows of 128 bytes apart
            uint32_t s = 0, phase = 0, g = 0, local = 0; // g: chunks so far, over all items
            for (int i = blockIdx.x; i < total; i += gridDim.x) {
                const MlpItem t = mlp_item<NT>(p, tiles, slices, s_off, s_pad, i);
                if (t.n == 0) continue;
                const uint32_t idesc1 = instr_desc(t.n, false, false), idesc2 = instr_desc(t.n, false, true);
                mbar_wait_lean(x_full, local & 1, dead, p.status);
                for (int c = 0; c <= t.chunks; ++c) {
                    if (c < t.chunks) {                  // GEMM1 of chunk c
                        const uint32_t gc = g + c, a = gc & 1;
                        mbar_wait_lean(&acc1_empty[a], ((gc >> 1) & 1) ^ 1, dead, p.status);
                        tc_fence_after();
                        for (int kb = 0; kb < KB1; ++kb) {
                            mbar_wait_lean(&full[s], phase, dead, p.status);
                            tc_fence_after();
                            const uint64_t da = d_ring + s * (BOX_BYTES >> 4), db = d_x + kb * (XKB_BYTES >> 4);
#pragma unroll
                            for (int kk = 0; kk < BK / UMMA_K; ++kk)
                                umma_bf16(tmem_base + a * NT, da + ((kk * UMMA_K * 2) >> 4), db + ((kk * UMMA_K * 2) >> 4), idesc1, (kb | kk) != 0);
                            umma_commit(&empty[s]);
                            if (++s == STAGES) { s = 0; phase ^= 1; }
                        }
                        umma_commit(&acc1_full[a]);
                        if (c == t.chunks - 1) umma_commit(x_empty);
                    }
                    if (c > 0) {                         // GEMM2 of chunk c - 1
                        const uint32_t gc = g + c - 1, a = gc & 1;
                        mbar_wait_lean(&act_full[a], (gc >> 1) & 1, dead, p.status);
                        if (c == 1) mbar_wait_lean(acc2_empty, (local & 1) ^ 1, dead, p.status);
                        tc_fence_after();
                        for (int m = 0; m < MT; ++m)
                            for (int kh = 0; kh < 2; ++kh) {
                                mbar_wait_lean(&full[s], phase, dead, p.status);
                                tc_fence_after();
                                const uint64_t da = d_ring + s * (BOX_BYTES >> 4), db = d_act + ((a * ACT_BYTES + kh * BK * 128) >> 4);
#pragma unroll
                                for (int kk = 0; kk < BK / UMMA_K; ++kk)
                                    umma_bf16(acc2_tmem + m * NT, da + ((kk * UMMA_K * 2) >> 4), db + ((kk * UMMA_K * 128) >> 4), idesc2,
                                              (c - 1) | kh | kk);
                                umma_commit(&empty[s]);
                                if (++s == STAGES) { s = 0; phase ^= 1; }
                            }
                        umma_commit(&act_empty[a]);
                    }
                }
                umma_commit(acc2_full);
                g += t.chunks;
                ++local;
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..17)
        const int quad = warp & 3, part = (warp - 2) >> 2;     // tensor-memory lanes 32 quad .., 16-token groups part, part + 4
        const uint32_t lanes = (uint32_t)(quad * 32) << 16;
        const int hid = quad * 32 + lane;                      // hidden unit of the chunk = contraction row of GEMM2
        uint32_t g = 0, local = 0;
        for (int i = blockIdx.x; i < total; i += gridDim.x) {
            const MlpItem t = mlp_item<NT>(p, tiles, slices, s_off, s_pad, i);
            if (t.n == 0) continue;
            // lane l keeps the slot of token 16 (part + 4 (l / 16)) + l % 16 of the tile, for the stores at the end
            const int tok = 16 * (part + 4 * (lane >> 4)) + (lane & 15);
            const int slot = tok < t.rows ? p.slot_of_prow[t.row0 + tok] : -1;
            for (int c = 0; c < t.chunks; ++c, ++g) {
                const uint32_t a = g & 1, ph = (g >> 1) & 1;
                const bool real = (t.c0 + c) * HC + hid < p.h;   // past the hidden width: the box held another expert's rows
                mbar_wait_lean(&acc1_full[a], ph, dead, p.status);
                tc_fence_after();
                uint32_t w[2][8];
#pragma unroll
                for (int q = 0; q < (NT > 64 ? 2 : 1); ++q) {
                    const int grp = part + 4 * q;
                    if (grp * 16 >= t.n) break;          // uniform
                    float v[16];
                    tmem_load_16_nowait(tmem_base + lanes + a * NT + grp * 16, (uint32_t*)v);
                    tmem_load_wait();
                    act_chunk_any<false, 16>(p.act, v, nullptr);
#pragma unroll
                    for (int j = 0; j < 8; ++j) w[q][j] = real ? pack_bf16(v[2 * j], v[2 * j + 1]) : 0u;
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc1_empty[a]);
                mbar_wait_lean(&act_empty[a], ph ^ 1, dead, p.status);       // GEMM2 two chunks back has read this buffer
#pragma unroll
                for (int q = 0; q < (NT > 64 ? 2 : 1); ++q) {
                    const int grp = part + 4 * q;
                    if (grp * 16 >= t.n) break;
                    uint8_t* row = s_act + a * ACT_BYTES + (grp >> 2) * (HC * 128) + hid * 128;
                    const int piece = 2 * (grp & 3), sw = hid & 7;           // 128-byte swizzle: piece j of row k sits at j ^ (k % 8)
                    st_shared_16B(row + ((piece ^ sw) << 4), w[q][0], w[q][1], w[q][2], w[q][3]);
                    st_shared_16B(row + (((piece + 1) ^ sw) << 4), w[q][4], w[q][5], w[q][6], w[q][7]);
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&act_full[a]);
            }
            mbar_wait_lean(acc2_full, local & 1, dead, p.status);
            tc_fence_after();
            float* out = (float*)p.out + (int64_t)t.slice * p.slots * p.r;
            for (int m = 0; m < MT; ++m) {
                const int col = m * 128 + hid;
#pragma unroll
                for (int q = 0; q < (NT > 64 ? 2 : 1); ++q) {
                    const int grp = part + 4 * q;
                    if (grp * 16 >= t.n) break;
                    float v[16];
                    tmem_load_16_nowait(acc2_tmem + lanes + m * NT + grp * 16, (uint32_t*)v);
                    tmem_load_wait();
                    if (slices > 1) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const int to = __shfl_sync(0xffffffffu, slot, 16 * q + j);
                            if (to >= 0 && col < p.r) out[(int64_t)to * p.r + col] = v[j];
                        }
                    } else {                             // neighbouring lanes swap halves of a token pair: an even lane has two columns
#pragma unroll                                           // of the first token, an odd lane of the second
                        for (int j = 0; j < 16; j += 2) {
                            const bool odd = lane & 1;
                            const float other = __shfl_xor_sync(0xffffffffu, odd ? v[j] : v[j + 1], 1);
                            const int to0 = __shfl_sync(0xffffffffu, slot, 16 * q + j), to1 = __shfl_sync(0xffffffffu, slot, 16 * q + j + 1);
                            const int to = odd ? to1 : to0;
                            const uint32_t w = odd ? pack_bf16(other, v[j + 1]) : pack_bf16(v[j], other);
                            if (to >= 0 && col < p.r) *(uint32_t*)((__nv_bfloat16*)p.out + (int64_t)to * p.r + (col & ~1)) = w;
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc2_empty);
            ++local;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

template <int NT, int STAGES>
cudaError_t launch(const CUtensorMap& mx, const CUtensorMap& m1, const CUtensorMap& m2, const MlpParams& p, cudaStream_t stream) {
    const size_t smem = (size_t)STAGES * BOX_BYTES + 2 * (size_t)(NT / 64) * HC * 128 + (size_t)(p.r / BK) * NT * BK * 2 +
                        (2 * STAGES + 12) * 8 + 16 + (size_t)(p.E + 1) * 4 + p.E + 1024;
    if (smem > 232448) return cudaErrorInvalidConfiguration;
    static PerDeviceOnce once;
    int dev;
    if (once.needed(&dev)) {
        cudaError_t e = cudaFuncSetAttribute(fused_mlp_kernel<NT, STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
        if (e != cudaSuccess) return e;
        once.mark(dev);
    }
    const int64_t items = (int64_t)p.max_tiles * (128 / NT) * p.sl.most;
    return launch_chained(fused_mlp_kernel<NT, STAGES>, (unsigned)(items < sm_count() ? items : sm_count()), kMlpThreads, smem, stream, mx, m1, m2, p);
}

}  // namespace

bool fused_mlp_supported(int r, int h, int dtype) {
    return dtype == BIGMAC_BF16 && r >= 64 && r <= 512 && r % 64 == 0 && h >= 64 && h % 64 == 0;
}

MlpSlicing fused_mlp_slicing(int r, int h, int64_t N, int64_t P) { return mlp_slicing(sm_count(), r, h, N, P); }

// xg [max_rows, r] grouped padded rows, w1 [E, h, r], w2 [E, r, h], out [slices][slots][r]; tiles of 128 rows and the tables
// on the device.
cudaError_t launch_fused_mlp(const void* xg, const void* w1, const void* w2, void* out, int64_t max_rows, int64_t slots,
                             const MlpSlicing& sl, int r, int h, int E, int act, const Tables& tb, int* status, cudaStream_t stream) {
    if (max_rows < kPad) return cudaSuccess;
    CUtensorMap mx, m1, m2;
    bool ok = make_map(&mx, xg, (uint64_t)r, (uint64_t)max_rows, (uint64_t)r, BK, 16);
    ok &= make_map(&m1, w1, (uint64_t)r, (uint64_t)E * h, (uint64_t)r, BK, 128);
    ok &= make_map(&m2, w2, (uint64_t)h, (uint64_t)E * r, (uint64_t)h, BK, 128);
    if (!ok) return cudaErrorInvalidValue;
    MlpParams p{};
    p.out = out; p.E = E; p.slots = slots; p.r = r; p.h = h; p.act = act; p.sl = sl;
    p.poffsets = tb.poffsets; p.counts = tb.counts; p.slot_of_prow = tb.slot_of_prow;
    p.max_tiles = (int)(max_rows / kPad); p.status = status;
    // the tables of more than 300 experts take the place of a stage
    if (r <= 256) return E <= 300 ? launch<128, 6>(mx, m1, m2, p, stream) : launch<128, 5>(mx, m1, m2, p, stream);
    return E <= 300 ? launch<64, 8>(mx, m1, m2, p, stream) : launch<64, 7>(mx, m1, m2, p, stream);
}

}  // namespace bigmac
