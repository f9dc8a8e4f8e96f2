// Both contractions of an expert in one kernel on CTA pairs, for every row of its segment: the training forward
//     z = x W1_e^T,  a = sigma(z),  u = a W2_e^T          (a and sigma'(z) are written for the backward),
// the inference forward (only u is written), and the input half of the backward
//     dz = (du W2_e) sigma'(z),  dxg = dz W1_e            (dz is written for the weight gradient).
// The matrix in the middle, by far the widest, goes from one contraction into the other through shared memory and is not
// read back from memory; as two launches the second one reads it again and all of its rows wait for all of the first.
//
// A work item is a pair of 128-row tiles of one expert; CTA r of the pair owns rows 128 r.. .  It walks the hidden width in
// chunks of 128 columns:
//   A(c)    acc1[c % 2] (128 rows x 128, tensor memory of each CTA) = X B1[chunk]^T          K = r, M = 256, N = 128
//   middle  eight epilogue warps, one group for even and one for odd chunks, read acc1, apply the activation (or multiply by
//           the saved sigma') and write bf16 to mid[c % 2], two 64-column blocks in the 128-byte swizzle: at once the K-major
//           A operand of the next contraction and the box of a TMA store
//   B(c)    acc2 (128 rows x r) += mid[c % 2] B2[chunk]                                      K = 128, M = 256, N = r
// The issuer runs A two chunks ahead of B, across the ends of items too (a group's next accumulator is then ready when it has
// written its chunk), but issues the first two As of an item behind the B of their turn, so that the rows X of the item, whose place
// the last A of the item before frees, have two chunks' time to arrive; acc2 is read out beside the first chunks of the next item.  Every SM stages half of each B
// (cta_group::2).  An extra thread moves the middle to memory (TMA stores of 128-row boxes).  sigma' goes from registers to
// memory and back in an order of its own, which only this kernel knows: the bytes of (row tile, chunk, warp) in the order of
// the warp's 16-byte accesses.
//
// What bounds it: the epilogue warps beside the writing of the middle.  d 2048 r 256 h 1024, 3001 tokens, cycles a chunk of 128 columns (ncu, active
// cycles over the chunks of a pair): 4900 training forward, 4300 backward, 3650 inference, of which the MMAs need 2050; clock stamps of an
// earlier build had 3200 forward without the stores, 2750 without arithmetic either.  131072 rows forward write 0.40 GB (103 us at the
// 3.9 TB/s this part writes at) in 190 us under the power cap (as two launches 133 + 78), backward 168 (99 + 78).
// Measured on the way there (3001 tokens' experts, inference / training forward, us): all sixteen warps on every chunk, A one
// ahead 54 / 64; two groups 48 / 59; A two ahead 44 / 59; sigma' past shared memory, whose place the ring takes 43 / 53.
#include "tc_pair.cuh"

namespace bigmac {

using namespace tc;

namespace {

enum FfnMode { FFN_TRAIN = 0, FFN_BWD = 1, FFN_INFER = 2 };

constexpr int HC = 128;                                  // hidden columns per chunk
constexpr uint32_t kStageBytes = 16384;                  // ring stage: 16 KB of B1 (two k slices of 64 columns) or of B2 (a k slice)
constexpr uint32_t kSliceBytes = 8192;                   // 64 x 64 bf16
constexpr uint32_t kMidBytes = 128 * HC * 2;
constexpr int kFfnThreads = (2 + kEpiWarps + 1) * 32;

struct FfnParams {
    __nv_bfloat16* out;      // [rows, r]
    uint8_t* sigma;          // [rows / 128][h / 128][16 KB]
    int r, h, act, E;
    const int32_t* poffsets;
    int* status;
};

struct FfnItem { int expert, m0, halves; };

__device__ __forceinline__ FfnItem ffn_item(const FfnParams& p, const int32_t* s_pp, int i) {
    int lo = 0, hi = p.E;                                // largest expert whose pairs begin at or before i
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (s_pp[mid] <= i) lo = mid; else hi = mid;
    }
    const int32_t* s_off = s_pp + p.E + 1;
    const int j = i - s_pp[lo];
    FfnItem t;
    t.expert = lo;
    t.m0 = s_off[lo] + 2 * j * BM;
    t.halves = min(2, (s_off[lo + 1] - s_off[lo]) / BM - 2 * j);
    return t;
}

// The chunks of a pair's items in order.
struct FfnWalk {
    int i, c, n;             // item, chunk of it, number of the item along the walk
    FfnItem t;
    __device__ __forceinline__ void begin(const FfnParams& p, const int32_t* s_pp, int first, int total) {
        i = first; c = 0; n = 0;
        if (i < total) t = ffn_item(p, s_pp, i);
    }
    __device__ __forceinline__ void next(const FfnParams& p, const int32_t* s_pp, int chunks, int stride, int total) {
        if (++c < chunks) return;
        c = 0; ++n; i += stride;
        if (i < total) t = ffn_item(p, s_pp, i);
    }
};

__device__ __forceinline__ void mbar_arrive_release_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

template <int MODE, int STAGES, bool GELU>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kFfnThreads, 1)
ffn_pair_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_b1,
                const __grid_constant__ CUtensorMap map_b2, const __grid_constant__ CUtensorMap map_mid, const FfnParams p) {
    constexpr bool BWD = MODE == FFN_BWD, STORES = MODE != FFN_INFER;
    const int KB = p.r / BK;                             // k slices of A: 2 or 4
    const int chunks = p.h / HC;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* s_ring = smem;
    uint8_t* s_mid = s_ring + STAGES * kStageBytes;      // [2]
    uint8_t* s_x = s_mid + 2 * kMidBytes;                // KB slices of 128 rows x 64
    uint64_t* full = (uint64_t*)(s_x + (uint32_t)KB * (BM * BK * 2));
    uint64_t* empty = full + STAGES;
    uint64_t* x_full = empty + STAGES;       uint64_t* x_empty = x_full + 1;
    uint64_t* acc1_full = x_full + 2;        uint64_t* acc1_empty = x_full + 4;      // [2] each
    uint64_t* mid_full = x_full + 6;         uint64_t* mid_empty = x_full + 8;       // [2] each; mid_full: the leader's, both CTAs arrive
    uint64_t* mid_here = x_full + 10;        // [2] this CTA's half is written (for the store)
    uint64_t* acc2_full = x_full + 12;       uint64_t* acc2_empty = x_full + 13;
    uint32_t* tmem_slot = (uint32_t*)(x_full + 14);
    volatile int* dead = (volatile int*)(tmem_slot + 1);
    int32_t* s_pp = (int32_t*)(tmem_slot + 4);           // [E + 1] pairs before an expert, [E + 1] padded offsets

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const bool leader = rank == 0;
    if (threadIdx.x == 32) {                             // the maps are on their way while the barriers are set up
        prefetch_tensormap(&map_x);
        prefetch_tensormap(&map_b1);
        prefetch_tensormap(&map_b2);
        if (STORES) prefetch_tensormap(&map_mid);
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(x_full, 1); mbar_init(x_empty, 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(&acc1_full[s], 1); mbar_init(&acc1_empty[s], kEpiWarps);       // eight warps of either CTA
            mbar_init(&mid_full[s], kEpiWarps); mbar_init(&mid_empty[s], STORES ? 2 : 1);
            mbar_init(&mid_here[s], kEpiWarps / 2);
        }
        mbar_init(acc2_full, 1); mbar_init(acc2_empty, 2 * kEpiWarps);
        *dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc_pair(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                  // the peer's barriers exist before anything signals them
    // Chained launch: everything above touched no global memory and may have run while the kernel before this one in
    // the stream was still working.  Tensor memory is held, so the next kernel of the stream may be set up in turn;
    // from the wait on, the predecessor's results are complete.
    grid_dependency_launch();
    grid_dependency_wait();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot, acc2_tmem = tmem_base + 2 * HC;
    int32_t* s_off = s_pp + p.E + 1;
    for (int e = threadIdx.x; e <= p.E; e += kFfnThreads) s_off[e] = p.poffsets[e];
    __syncthreads();
    if (warp == 0) warp_prefix(p.E, s_pp, [&](int e) { return ((s_off[e + 1] - s_off[e]) / kPad + 1) / 2; });
    __syncthreads();
    const int total = s_pp[p.E], first = blockIdx.x >> 1, stride = gridDim.x >> 1;

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer (both CTAs)
        if (elect_one()) {
            uint32_t s = 0, phase = 1;
            const uint32_t leader_full = map_to_cta(full, 0), leader_x = map_to_cta(x_full, 0);
            const int half_r = p.r / 2;
            auto b1 = [&](const FfnItem& t, int c) {     // this CTA's 64 hidden columns of chunk c, two k slices a stage
                for (int kb = 0; kb < KB; kb += 2) {
                    mbar_wait_lean(&empty[s], phase, dead, p.status);
                    if (leader) mbar_expect_tx(&full[s], 4 * kSliceBytes);
                    const int n0 = c * HC + (int)rank * 64;
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        uint8_t* dst = s_ring + s * kStageBytes + q * kSliceBytes;
                        if (BWD) tma_load_2d_pair(dst, &map_b1, leader_full + 8 * s, n0, t.expert * p.r + (kb + q) * BK);
                        else tma_load_2d_pair(dst, &map_b1, leader_full + 8 * s, (kb + q) * BK, t.expert * p.h + n0);
                    }
                    if (++s == STAGES) { s = 0; phase ^= 1; }
                }
            };
            auto b2 = [&](const FfnItem& t, int c) {     // this CTA's r / 2 columns of u (dxg), a k slice a stage
                for (int kh = 0; kh < 2; ++kh) {
                    mbar_wait_lean(&empty[s], phase, dead, p.status);
                    if (leader) mbar_expect_tx(&full[s], (uint32_t)(2 * half_r * BK * 2));
                    uint8_t* dst = s_ring + s * kStageBytes;
                    const int k0 = c * HC + kh * BK, n0 = (int)rank * half_r;
                    if (BWD) {
                        for (int q = 0; q < half_r; q += 64)
                            tma_load_2d_pair(dst + q / 64 * kSliceBytes, &map_b2, leader_full + 8 * s, n0 + q, t.expert * p.h + k0);
                    } else {
                        tma_load_2d_pair(dst, &map_b2, leader_full + 8 * s, k0, t.expert * p.r + n0);
                    }
                    if (++s == STAGES) { s = 0; phase ^= 1; }
                }
            };
            FfnWalk wa, wb;
            wa.begin(p, s_pp, first, total);
            wb = wa;
            auto next_a = [&]() {                        // in the order of the MMAs
                if (wa.i >= total) return;
                if (wa.c == 0) {
                    mbar_wait_lean(x_empty, (wa.n & 1) ^ 1, dead, p.status);
                    if (leader) mbar_expect_tx(x_full, (uint32_t)(2 * KB * BM * BK * 2));
                    for (int kb = 0; kb < KB; ++kb) tma_load_2d_pair(s_x + kb * (BM * BK * 2), &map_x, leader_x, kb * BK, wa.t.m0 + (int)rank * BM);
                }
                b1(wa.t, wa.c);
                wa.next(p, s_pp, chunks, stride, total);
            };
            next_a();
            next_a();
            for (; wb.i < total; wb.next(p, s_pp, chunks, stride, total)) {
                const bool a_first = wa.c > 1;
                if (a_first) next_a();
                b2(wb.t, wb.c);
                if (!a_first) next_a();
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (one thread of the leader CTA)
        if (leader && elect_one()) {
            constexpr uint32_t idesc1 = instr_desc_pair(HC, false, BWD);
            const uint32_t idesc2 = instr_desc_pair(p.r, false, BWD);
            // B K-major: rows of 128 bytes, a k step 32 bytes on; MN-major: 64-column blocks, a k step 16 rows of 128 bytes on
            const uint64_t d_x = smem_desc(smem_u32(s_x), 16, 1024), d_mid = smem_desc(smem_u32(s_mid), 16, 1024);
            const uint64_t d_ring = BWD ? smem_desc(smem_u32(s_ring), kSliceBytes, 1024) : smem_desc(smem_u32(s_ring), 16, 1024);
            constexpr uint32_t kStepA = (UMMA_K * 2) >> 4, kStepB = (BWD ? UMMA_K * 128 : UMMA_K * 2) >> 4;
            uint32_t s = 0, phase = 0;
            const int items = first < total ? (total - first + stride - 1) / stride : 0, all = items * chunks;
            int ga = 0, ca = 0, na = 0;                  // next A: its number, chunk and item
            auto contract_a = [&]() {
                if (ga == all) return;
                const uint32_t a = ga & 1;
                if (ca == 0) mbar_wait_lean(x_full, na & 1, dead, p.status);
                mbar_wait_lean(&acc1_empty[a], ((ga >> 1) & 1) ^ 1, dead, p.status);
                tc_fence_after();
                for (int kb = 0; kb < KB; kb += 2) {
                    mbar_wait_lean(&full[s], phase, dead, p.status);
                    tc_fence_after();
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const uint64_t da = d_x + (kb + q) * ((BM * BK * 2) >> 4), db = d_ring + ((s * kStageBytes + q * kSliceBytes) >> 4);
#pragma unroll
                        for (int kk = 0; kk < BK / UMMA_K; ++kk)
                            umma_bf16_pair(tmem_base + a * HC, da + kk * kStepA, db + kk * kStepB, idesc1, (kb | q | kk) != 0);
                    }
                    umma_commit_pair(&empty[s]);
                    if (++s == STAGES) { s = 0; phase ^= 1; }
                }
                umma_commit_pair(&acc1_full[a]);
                ++ga;
                if (++ca == chunks) { umma_commit_pair(x_empty); ca = 0; ++na; }
            };
            contract_a();
            contract_a();
            for (int gb = 0, cb = 0, nb = 0; gb < all; ++gb) {
                const bool a_first = ca > 1;
                if (a_first) contract_a();               // its accumulator is free before the middle that B waits for is written
                const uint32_t a = gb & 1;
                mbar_wait_cluster(&mid_full[a], (gb >> 1) & 1, dead, p.status);
                if (cb == 0) mbar_wait_lean(acc2_empty, (nb & 1) ^ 1, dead, p.status);
                fence_async_smem();
                tc_fence_after();
                for (int kh = 0; kh < 2; ++kh) {
                    mbar_wait_lean(&full[s], phase, dead, p.status);
                    tc_fence_after();
                    const uint64_t da = d_mid + ((a * kMidBytes + kh * (kMidBytes / 2)) >> 4), db = d_ring + s * (kStageBytes >> 4);
#pragma unroll
                    for (int kk = 0; kk < BK / UMMA_K; ++kk)
                        umma_bf16_pair(acc2_tmem, da + kk * kStepA, db + kk * kStepB, idesc2, (cb | kh | kk) != 0);
                    umma_commit_pair(&empty[s]);
                    if (++s == STAGES) { s = 0; phase ^= 1; }
                }
                umma_commit_pair(&mid_empty[a]);
                if (++cb == chunks) { umma_commit_pair(acc2_full); cb = 0; ++nb; }
                if (!a_first) contract_a();
            }
        }
    } else if (warp == 2 + kEpiWarps) {
        // ------------------------------------------------------------------ the middle to memory (one thread)
        if (STORES && elect_one()) {
            FfnWalk w;
            w.begin(p, s_pp, first, total);
            for (uint32_t g = 0; w.i < total; ++g, w.next(p, s_pp, chunks, stride, total)) {
                const uint32_t a = g & 1, ph = (g >> 1) & 1;
                mbar_wait_lean(&mid_here[a], ph, dead, p.status);
                if ((int)rank < w.t.halves) {            // else the rows are another expert's
                    const int row0 = w.t.m0 + (int)rank * BM;
                    tma_store_2d(&map_mid, s_mid + a * kMidBytes, w.c * HC, row0);
                    tma_store_2d(&map_mid, s_mid + a * kMidBytes + kMidBytes / 2, w.c * HC + 64, row0);
                    tma_store_commit();
                    tma_store_wait_read();
                }
                mbar_arrive(&mid_empty[a]);
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..17, both CTAs)
        const int quad = warp & 3, part = (warp - 2) >> 2;     // rows 32 quad ..
        const int group = part >> 1, half = part & 1;          // chunks of this parity, columns 64 half ..
        const uint32_t lanes = (uint32_t)(quad * 32) << 16, a = group;
        const int row = quad * 32 + lane, sw = row & 7;
        const uint32_t leader_acc1_empty = map_to_cta(&acc1_empty[a], 0), leader_mid_full = map_to_cta(&mid_full[a], 0), leader_acc2_empty = map_to_cta(acc2_empty, 0);
        uint8_t* mid_row = s_mid + a * kMidBytes + half * (kMidBytes / 2) + row * 128;
        uint4* sigma_here = (uint4*)(p.sigma + (half * 8 + quad) * 1024) + lane;       // + a tile's and a chunk's place; 32 columns on: 256
        auto sigma_at = [&](const FfnWalk& q) { return sigma_here + ((int64_t)(q.t.m0 / BM + (int)rank) * chunks + q.c) * (128 * HC / 16); };
        auto read_out = [&](int item) {                  // acc2 to memory, both groups
            const FfnItem t = ffn_item(p, s_pp, first + item * stride);
            mbar_wait_lean(acc2_full, item & 1, dead, p.status);
            tc_fence_after();
            const bool mine = (int)rank < t.halves;
            __nv_bfloat16* to = p.out + (int64_t)(t.m0 + (int)rank * BM + row) * p.r;
            for (int c0 = part * 32; c0 < p.r; c0 += 128) {
                float v[32];
                tmem_load_32(acc2_tmem + lanes + c0, (uint32_t*)v);
                if (c0 + 128 >= p.r) {                   // all of this warp's columns are read
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(leader_acc2_empty);
                }
                if (mine) {
                    uint32_t w[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) w[j] = pack_bf16(v[2 * j], v[2 * j + 1]);
                    st_global_32B(to + c0, w);
                    st_global_32B(to + c0 + 16, w + 8);
                }
            }
        };
        FfnWalk w;
        w.begin(p, s_pp, first, total);
        if (group == 1 && w.i < total) w.next(p, s_pp, chunks, stride, total);
        uint32_t zw[2][8];                               // BWD: sigma' of the group's next chunk
        auto fetch_z = [&](const FfnWalk& q, int half_chunk) {
            if (q.i >= total || (int)rank >= q.t.halves) return;
            const uint4* from = sigma_at(q) + half_chunk * 256;
            *(uint4*)zw[half_chunk] = __ldcs(from);
            *(uint4*)(zw[half_chunk] + 4) = __ldcs(from + 32);
        };
        if (BWD) { fetch_z(w, 0); fetch_z(w, 1); }
        int read = 0;                                    // items whose acc2 this warp has read out
        for (uint32_t ph = 0; w.i < total; ph ^= 1) {
            // The group with the first chunk of an item does that before it reads the item before out, the other one after:
            // acc2 is complete about when the first one has done its chunk.
            if (w.c > 0)
                while (read < w.n) read_out(read++);
            FfnWalk after = w;                           // the group's next chunk
            after.next(p, s_pp, chunks, stride, total);
            if (after.i < total) after.next(p, s_pp, chunks, stride, total);
            mbar_wait_lean(&acc1_full[a], ph, dead, p.status);
            tc_fence_after();
#pragma unroll (BWD ? 2 : 1)
            for (int q = 0; q < 2; ++q) {                // 32 columns
                float v[32];
                tmem_load_32(tmem_base + lanes + a * HC + half * 64 + q * 32, (uint32_t*)v);
                if (q == 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(leader_acc1_empty);
                }
                uint32_t o[16], wz[8];
                if (BWD) {
                    mul_by_sig32(v, zw[q]);
                    fetch_z(after, q);
                } else if (GELU) {
                    act_chunk<BIGMAC_ACT_GELU_ERF, STORES>(v, wz);
                } else {
                    act_chunk_any<STORES>(p.act, v, wz);
                }
#pragma unroll
                for (int j = 0; j < 16; ++j) o[j] = pack_bf16(v[2 * j], v[2 * j + 1]);
                if (q == 0) mbar_wait_lean(&mid_empty[a], ph ^ 1, dead, p.status);   // the group's chunk before is contracted and stored
#pragma unroll
                for (int j = 0; j < 4; ++j)              // 128-byte swizzle: piece j of a row sits at j ^ (row % 8)
                    st_shared_16B(mid_row + (((4 * q + j) ^ sw) << 4), o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
                if (MODE == FFN_TRAIN && (int)rank < w.t.halves) {
                    uint4* to = sigma_at(w) + q * 256;
                    __stcs(to, make_uint4(wz[0], wz[1], wz[2], wz[3]));
                    __stcs(to + 32, make_uint4(wz[4], wz[5], wz[6], wz[7]));
                }
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive_release_cluster(leader_mid_full);
                if (STORES) mbar_arrive(&mid_here[a]);
            }
            if (w.c == 0)
                while (read < w.n) read_out(read++);
            w = after;
        }
        for (const int items = first < total ? (total - first + stride - 1) / stride : 0; read < items;) read_out(read++);
    }
    if (STORES && warp == 2 + kEpiWarps && elect_one()) tma_store_wait_read();     // the boxes have left shared memory
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                  // nobody leaves while the peer may still touch this CTA
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, 512);
    }
}

template <int MODE, int STAGES, bool GELU>
cudaError_t launch(const CUtensorMap& mx, const CUtensorMap& m1, const CUtensorMap& m2, const CUtensorMap& mm, const FfnParams& p,
                   int64_t max_pairs, cudaStream_t stream) {
    constexpr size_t kMaxSmem = 232448;
    const size_t smem = STAGES * kStageBytes + 2 * kMidBytes + (size_t)(p.r / BK) * BM * BK * 2 + (2 * STAGES + 14) * 8 + 16 +
                        2 * (size_t)(p.E + 1) * 4 + 1024;
    if (smem > kMaxSmem) return cudaErrorInvalidConfiguration;
    static PerDeviceOnce once;
    int dev;
    if (once.needed(&dev)) {
        cudaError_t e = cudaFuncSetAttribute(ffn_pair_kernel<MODE, STAGES, GELU>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
        if (e != cudaSuccess) return e;
        once.mark(dev);
    }
    int64_t clusters = sm_count() / 2;
    if (max_pairs < clusters) clusters = max_pairs;
    if (clusters < 1) clusters = 1;
    return launch_chained(ffn_pair_kernel<MODE, STAGES, GELU>, (unsigned)(2 * clusters), kFfnThreads, smem, stream, mx, m1, m2, mm, p);
}

template <int MODE, bool GELU>
cudaError_t run(const void* x, const void* b1, const void* b2, void* mid, void* sigma, void* out, int64_t max_rows, int r, int h, int E,
                int act, const int32_t* poffsets, int* status, cudaStream_t stream) {
    CUtensorMap mx, m1, m2;
    bool ok = make_map(&mx, x, (uint64_t)r, (uint64_t)max_rows, (uint64_t)r, BK, BM);
    if (MODE == FFN_BWD) {                               // B1 = W2_e [r, h], B2 = W1_e [h, r], both read along their rows
        ok &= make_map(&m1, b1, (uint64_t)h, (uint64_t)E * r, (uint64_t)h, 64, BK);
        ok &= make_map(&m2, b2, (uint64_t)r, (uint64_t)E * h, (uint64_t)r, 64, BK);
    } else {                                             // B1 = W1_e [h, r], B2 = W2_e [r, h]: K-major
        ok &= make_map(&m1, b1, (uint64_t)r, (uint64_t)E * h, (uint64_t)r, BK, 64);
        ok &= make_map(&m2, b2, (uint64_t)h, (uint64_t)E * r, (uint64_t)h, BK, (uint32_t)(r / 2));
    }
    CUtensorMap mm = mx;
    if (MODE != FFN_INFER) ok &= make_map(&mm, mid, (uint64_t)h, (uint64_t)max_rows, (uint64_t)h, 64, BM);
    if (!ok) return cudaErrorInvalidValue;
    FfnParams p{};
    p.out = (__nv_bfloat16*)out; p.sigma = (uint8_t*)sigma; p.r = r; p.h = h; p.act = act; p.E = E; p.poffsets = poffsets; p.status = status;
    const int64_t pairs = (max_rows / BM + 1) / 2 + E;   // at most: the kernel counts them from the offsets
    // as many stages as there is room for; the tables of more than 200 experts take the place of one
    if (r == 256) return E <= 200 ? launch<MODE, 6, GELU>(mx, m1, m2, mm, p, pairs, stream) : launch<MODE, 5, GELU>(mx, m1, m2, mm, p, pairs, stream);
    return launch<MODE, 7, GELU>(mx, m1, m2, mm, p, pairs, stream);
}

}  // namespace

bool ffn_pair_supported(int r, int h, int E, int dtype) {
    return dtype == BIGMAC_BF16 && (r == 128 || r == 256) && h % HC == 0 && E <= kMaxExperts;
}

cudaError_t launch_ffn_forward(const void* xg, const void* w1, const void* w2, void* a, void* sigma, void* u, int64_t max_rows, int r, int h,
                               int E, int act, const int32_t* poffsets, int* status, cudaStream_t stream) {
    if (max_rows < kPad) return cudaSuccess;
    const bool gelu = act == BIGMAC_ACT_GELU_ERF;
    if (sigma)
        return gelu ? run<FFN_TRAIN, true>(xg, w1, w2, a, sigma, u, max_rows, r, h, E, act, poffsets, status, stream)
                    : run<FFN_TRAIN, false>(xg, w1, w2, a, sigma, u, max_rows, r, h, E, act, poffsets, status, stream);
    return gelu ? run<FFN_INFER, true>(xg, w1, w2, nullptr, nullptr, u, max_rows, r, h, E, act, poffsets, status, stream)
                : run<FFN_INFER, false>(xg, w1, w2, nullptr, nullptr, u, max_rows, r, h, E, act, poffsets, status, stream);
}

cudaError_t launch_ffn_backward(const void* du, const void* w1, const void* w2, void* dz, const void* sigma, void* dxg, int64_t max_rows, int r,
                                int h, int E, const int32_t* poffsets, int* status, cudaStream_t stream) {
    if (max_rows < kPad) return cudaSuccess;
    return run<FFN_BWD, false>(du, w2, w1, dz, const_cast<void*>(sigma), dxg, max_rows, r, h, E, 0, poffsets, status, stream);
}

}  // namespace bigmac
