// Row-move kernels of the exchange stage: dispatch (token rows -> expert-grouped rows), combine
// (gate-weighted return to token order) and their backward twins.  All rows move as 16-byte vectors;
// one warp owns one destination row, so every output element is written once and summed in a fixed
// order (deterministic, no atomics).
#include "internal.h"

namespace bigmac {

namespace {

constexpr unsigned kFull = 0xffffffffu;

template <typename T> struct Vec;          // 16 bytes of T
template <> struct Vec<float> {
    static constexpr int kElems = 4;
    static __device__ __forceinline__ void unpack(const uint4& v, float* f) {
        f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y); f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
    }
    static __device__ __forceinline__ uint4 pack(const float* f) {
        return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
    }
};
template <> struct Vec<__nv_bfloat16> {
    static constexpr int kElems = 8;
    static __device__ __forceinline__ void unpack(const uint4& v, float* f) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f[2 * i] = __uint_as_float(w[i] << 16);
            f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
    static __device__ __forceinline__ uint4 pack(const float* f) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            __nv_bfloat162 p = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
            w[i] = *reinterpret_cast<uint32_t*>(&p);
        }
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
};

__device__ __forceinline__ int warp_global_id() { return blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); }

// Each warp moves kDispatchRows consecutive grouped rows: all row indices are read first, then every
// 16-byte load of the rows is issued before the first store, so many loads are in flight per lane.
constexpr int kDispatchRows = 4;
__global__ void __launch_bounds__(256) dispatch_kernel(const uint4* __restrict__ src, uint4* __restrict__ grouped,
                                                       const int32_t* __restrict__ slot_of_prow,
                                                       const int32_t* __restrict__ n_tiles, int k, int vecs_per_row,
                                                       int64_t max_prows) {
    grid_dependency_wait();
    grid_dependency_launch();
    const int64_t prow0 = (int64_t)warp_global_id() * kDispatchRows;
    int64_t live = (int64_t)(*n_tiles) * kPad;              // a multiple of kDispatchRows
    if (live > max_prows) live = max_prows;
    if (prow0 >= live) return;
    const int lane = threadIdx.x & 31;
    int s[kDispatchRows];
#pragma unroll
    for (int i = 0; i < kDispatchRows; ++i) s[i] = slot_of_prow[prow0 + i];
    for (int c0 = 0; c0 < vecs_per_row; c0 += 64) {
        uint4 v[kDispatchRows][2];
#pragma unroll
        for (int i = 0; i < kDispatchRows; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int c = c0 + lane + 32 * j;
                v[i][j] = (s[i] >= 0 && c < vecs_per_row) ? src[(int64_t)(s[i] / k) * vecs_per_row + c] : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
        for (int i = 0; i < kDispatchRows; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int c = c0 + lane + 32 * j;
                if (c < vecs_per_row) grouped[(prow0 + i) * vecs_per_row + c] = v[i][j];
            }
    }
}

// A warp per token.  The rows of eight slots are fetched together (lane j reads the place and weight of slot j, all row
// loads of a batch are issued before the first is used), then added in slot order: with one dependent load per slot the
// kernel waited for eight round trips to L2 in a row.  MAY_DROP: slots may carry row -1 (dropped under a capacity limit)
// and are then left out.
template <typename T, bool MAY_DROP>
__global__ void __launch_bounds__(256) combine_kernel(const uint4* __restrict__ grouped, uint4* __restrict__ dst,
                                                      const float* __restrict__ w,
                                                      const int32_t* __restrict__ prow_of_slot, int n_tokens, int k,
                                                      int vecs_per_row, int dst_vecs_per_row) {
    grid_dependency_wait();
    grid_dependency_launch();
    constexpr int V = Vec<T>::kElems, B = 8;
    const int t = warp_global_id();
    if (t >= n_tokens) return;
    const int lane = threadIdx.x & 31;
    for (int c0 = 0; c0 < vecs_per_row; c0 += 32) {
        const int c = c0 + lane;
        const bool mine = c < vecs_per_row;
        float acc[V];
#pragma unroll
        for (int i = 0; i < V; ++i) acc[i] = 0.0f;
        for (int j0 = 0; j0 < k; j0 += B) {
            int place = -1;
            float weight = 1.0f;
            if (lane < B && j0 + lane < k) {
                const int64_t s = (int64_t)t * k + j0 + lane;
                place = prow_of_slot[s];
                if (!MAY_DROP) place = max(place, 0);        // dropless rows are never negative; keeps the address in range if one were
                if (w) weight = w[s];
            }
            uint4 v[B];
#pragma unroll
            for (int j = 0; j < B; ++j) {
                const int prow = __shfl_sync(kFull, place, j);
                v[j] = (mine && prow >= 0) ? grouped[(int64_t)prow * vecs_per_row + c] : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int j = 0; j < B; ++j) {                      // slot order: fixed summation order
                if (__shfl_sync(kFull, place, j) < 0) continue;
                const float p = __shfl_sync(kFull, weight, j);
                float f[V];
                Vec<T>::unpack(v[j], f);
#pragma unroll
                for (int i = 0; i < V; ++i) acc[i] = fmaf(p, f[i], acc[i]);
            }
        }
        if (mine) dst[(int64_t)t * dst_vecs_per_row + c] = Vec<T>::pack(acc);
    }
}

// Combine of the fused expert kernel's fp32 rows, [parts][T k][r]: the rows of a token's slots lie side by side, a thread
// owns four columns of one token.  The loads of eight slots of one slice are in flight together.
template <bool MAY_DROP>
__global__ void __launch_bounds__(128) combine_parts_kernel(const float4* __restrict__ src, const int32_t* __restrict__ n_tiles,
                                                            MlpSlicing sl, int64_t part_stride, uint2* __restrict__ dst,
                                                            const float* __restrict__ w, const int32_t* __restrict__ prow_of_slot,
                                                            int T, int k, int quads) {
    grid_dependency_wait();
    grid_dependency_launch();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)T * quads) return;
    const int parts = mlp_slices(sl, *n_tiles);
    const int64_t t = i / quads;
    const int c = (int)(i - t * quads);
    float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float4* row = src + t * k * quads + c;
    for (int j0 = 0; j0 < k; j0 += 8) {
        float4 u[8];
        float p[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            p[j] = j0 + j < k ? w[t * k + j0 + j] : 0.0f;
            if (MAY_DROP && j0 + j < k && prow_of_slot[t * k + j0 + j] < 0) p[j] = 0.0f;
            u[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        if (parts == 1) {                                // bf16 rows
            uint2 v[8];
            const uint2* from = reinterpret_cast<const uint2*>(src) + t * k * quads + c;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bool there = j0 + j < k && (!MAY_DROP || prow_of_slot[t * k + j0 + j] >= 0);
                v[j] = there ? from[(int64_t)(j0 + j) * quads] : make_uint2(0, 0);
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
                u[j] = make_float4(__uint_as_float(v[j].x << 16), __uint_as_float(v[j].x & 0xffff0000u), __uint_as_float(v[j].y << 16),
                                   __uint_as_float(v[j].y & 0xffff0000u));
        }
        else for (int s = 0; s < parts; ++s) {           // slices in order inside a slot
            float4 v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bool there = j0 + j < k && (!MAY_DROP || prow_of_slot[t * k + j0 + j] >= 0);
                v[j] = there ? row[s * part_stride + (int64_t)(j0 + j) * quads] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) { u[j].x += v[j].x; u[j].y += v[j].y; u[j].z += v[j].z; u[j].w += v[j].w; }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {                    // slot order
            acc.x = fmaf(p[j], u[j].x, acc.x); acc.y = fmaf(p[j], u[j].y, acc.y); acc.z = fmaf(p[j], u[j].z, acc.z); acc.w = fmaf(p[j], u[j].w, acc.w);
        }
    }
    const __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y), hi = __floats2bfloat162_rn(acc.z, acc.w);
    dst[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}

// Sums each of eight values over the warp's lanes: lane 4 j .. 4 j + 3 get the total of v[j] (v is used up).  Fixed order.
__device__ __forceinline__ float warp_sum8(float* v) {
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int n = 4; n > 0; n >>= 1, off >>= 1) {
        const bool upper = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float send = upper ? v[i] : v[i + n], keep = upper ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(kFull, send, off);
        }
    }
    v[0] += __shfl_xor_sync(kFull, v[0], 2);
    return v[0] + __shfl_xor_sync(kFull, v[0], 1);
}

// Backward of the combine, and (dlogits non-null) of the softmax over the k gate values: a warp per token reads dy' once, the
// rows of u of eight slots together, writes their rows of du and knows all of the token's dp, from which the gate's gradient
// follows without another launch.  The blocks behind the tokens' write zeros to the experts' padding rows, a block an expert.
// A slot without a row (dropped under a capacity limit) counts with dp = 0.
// Bound by HBM (u read, du written).  A warp per grouped row before, with a chain of three dependent loads for one row, and a
// launch of its own for the gate: a training step of fp32, 256 tokens, 61.0 -> 59.8 us; d 1024, 4096 tokens 137.4 -> 136.3; d 2048,
// 2999 tokens 280 -> 277.
// B slots of a token at once, C pieces of 32 vectors of each: B = 8, C = 1; with one or two slots a token B = 2, C = 2 (20000 tokens, one
// slot, with the gate: r 512 31.2 us with B = 8, 21.8 so, r 256 22.9 and 18.3; as two kernels 27 and 23).
template <typename T, int B, int C>
__global__ void __launch_bounds__(256) combine_bwd_kernel(const uint4* __restrict__ dy_lo, const uint4* __restrict__ u,
                                                          uint4* __restrict__ du, float* __restrict__ dp,
                                                          const int32_t* __restrict__ prow_of_slot, const float* __restrict__ topk_w,
                                                          const int32_t* __restrict__ topk_idx, const int32_t* __restrict__ counts,
                                                          const int32_t* __restrict__ poffsets, T* __restrict__ dlogits, int n_tokens,
                                                          int k, int vecs_per_row, int E, int width, int ld) {
    grid_dependency_wait();
    grid_dependency_launch();
    constexpr int V = Vec<T>::kElems;
    const int lane = threadIdx.x & 31, token_blocks = (n_tokens + 7) / 8;
    if ((int)blockIdx.x >= token_blocks) {
        const int e = blockIdx.x - token_blocks;
        const int64_t first = ((int64_t)poffsets[e] + counts[e]) * vecs_per_row, last = (int64_t)poffsets[e + 1] * vecs_per_row;
        for (int64_t i = first + threadIdx.x; i < last; i += 256) du[i] = make_uint4(0, 0, 0, 0);
        return;
    }
    const int t = warp_global_id();
    if (t >= n_tokens) return;
    const int64_t s0 = (int64_t)t * k;
    T* row = dlogits ? dlogits + (int64_t)t * ld : nullptr;
    if (row)
        for (int e = lane; e < width; e += 32) row[e] = (T)0.0f;
    float mine = 0.0f, weight = 0.0f;                        // k <= B: lane j has the j-th slot's dp, weight and expert
    int expert = -1;
    for (int j0 = 0; j0 < k; j0 += B) {
        int place = -1;
        weight = 0.0f;
        if (lane < B && j0 + lane < k) {
            place = prow_of_slot[s0 + j0 + lane];
            weight = topk_w[s0 + j0 + lane];
            expert = topk_idx[s0 + j0 + lane];
        }
        float dot[B];
#pragma unroll
        for (int j = 0; j < B; ++j) dot[j] = 0.0f;
        for (int c0 = 0; c0 < vecs_per_row; c0 += 32 * C) {
            const uint4 none = make_uint4(0, 0, 0, 0);
            uint4 g[C], v[C][B];
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const int c = c0 + 32 * q + lane;
                g[q] = c < vecs_per_row ? dy_lo[(int64_t)t * vecs_per_row + c] : none;
#pragma unroll
                for (int j = 0; j < B; ++j) {
                    const int prow = __shfl_sync(kFull, place, j);
                    v[q][j] = c < vecs_per_row && prow >= 0 ? u[(int64_t)prow * vecs_per_row + c] : none;
                }
            }
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const int c = c0 + 32 * q + lane;
                float a[V];
                Vec<T>::unpack(g[q], a);
#pragma unroll
                for (int j = 0; j < B; ++j) {
                    const int prow = __shfl_sync(kFull, place, j);
                    if (prow < 0) continue;                  // uniform
                    const float p = __shfl_sync(kFull, weight, j);
                    float b[V], o[V];
                    Vec<T>::unpack(v[q][j], b);
#pragma unroll
                    for (int i = 0; i < V; ++i) { dot[j] = fmaf(a[i], b[i], dot[j]); o[i] = p * a[i]; }
                    if (c < vecs_per_row) du[(int64_t)prow * vecs_per_row + c] = Vec<T>::pack(o);
                }
            }
        }
        if (B == 8) {
            const float total = warp_sum8(dot);
            mine = __shfl_sync(kFull, total, 4 * (lane & 7));
        } else {                                             // the same order of additions
#pragma unroll
            for (int j = 0; j < B; ++j) {
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) dot[j] += __shfl_xor_sync(kFull, dot[j], off);
                if (lane == j) mine = dot[j];
            }
        }
        if (lane < B && j0 + lane < k) dp[s0 + j0 + lane] = mine;
    }
    if (!row) return;
    __syncwarp();                                            // the zeros, and other lanes' dp, are there
    float part = 0.0f;
    if (k <= B) part = fmaf(weight, mine, part);             // (weight 0 beyond k)
    else
        for (int j = lane; j < k; j += 32) part = fmaf(topk_w[s0 + j], dp[s0 + j], part);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(kFull, part, off);
    auto give = [&](int j, float w, float g, int e) {
        const float dl = w * (g - part);
        if ((unsigned)e < (unsigned)E) row[e] = (T)dl;
        dp[s0 + j] = dl;                                     // fp32 copy per slot, for the bias gradient
    };
    if (k <= B) {
        if (lane < k) give(lane, weight, mine, expert);
    } else {
        for (int j = lane; j < k; j += 32) give(j, topk_w[s0 + j], dp[s0 + j], topk_idx[s0 + j]);
    }
}

template <typename T>
__global__ void __launch_bounds__(256) gate_bwd_kernel(float* __restrict__ dp, const float* __restrict__ topk_w,
                                                       const int32_t* __restrict__ topk_idx, T* __restrict__ dlogits,
                                                       int n_tokens, int E, int width, int ld, int k) {
    grid_dependency_wait();
    grid_dependency_launch();
    const int t = warp_global_id();
    if (t >= n_tokens) return;
    const int lane = threadIdx.x & 31;
    const float* p = topk_w + (int64_t)t * k;
    float* g = dp + (int64_t)t * k;
    float part = 0.0f;
    for (int j = lane; j < k; j += 32) part = fmaf(p[j], g[j], part);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(kFull, part, off);
    T* row = dlogits + (int64_t)t * ld;
    for (int e = lane; e < width; e += 32) row[e] = (T)0.0f;
    __syncwarp();
    for (int j = lane; j < k; j += 32) {
        const float dl = p[j] * (g[j] - part);
        const int e = topk_idx[(int64_t)t * k + j];
        if ((unsigned)e < (unsigned)E) row[e] = (T)dl;
        g[j] = dl;                                   // fp32 copy per slot, for the bias gradient
    }
}

// Bias gradient db[e] = sum over slots routed to e of dl[slot], from the fp32 per-slot values, in two
// deterministic stages.  Block b owns a contiguous range of slots, its warps contiguous sub-ranges; a warp walks
// its range 32 slots at a time and lane l adds, in slot order, the values of the experts e with e % 32 == l into
// the warp's row of shared memory.  The block then adds its warps' rows in order.
__global__ void __launch_bounds__(256) colsum_slots_kernel(const float* __restrict__ dl, const int32_t* __restrict__ topk_idx,
                                                           float* __restrict__ partial, int64_t N, int E) {
    grid_dependency_wait();
    grid_dependency_launch();
    extern __shared__ float warp_acc[];              // [8][E]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < 8 * E; i += blockDim.x) warp_acc[i] = 0.0f;
    __syncthreads();
    const int64_t per_warp = ((N + (int64_t)gridDim.x * 8 - 1) / ((int64_t)gridDim.x * 8) + 31) / 32 * 32;
    const int64_t s0 = ((int64_t)blockIdx.x * 8 + warp) * per_warp;
    const int64_t s1 = s0 + per_warp < N ? s0 + per_warp : N;
    float* mine = warp_acc + warp * E;
    for (int64_t base = s0; base < s1; base += 32) {
        const int64_t s = base + lane;
        const int e = s < s1 ? topk_idx[s] : -1;
        const float v = s < s1 ? dl[s] : 0.0f;
#pragma unroll 8
        for (int i = 0; i < 32; ++i) {
            const int ei = __shfl_sync(kFull, e, i);
            const float vi = __shfl_sync(kFull, v, i);
            if (ei >= 0 && (ei & 31) == lane) mine[ei] += vi;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += blockDim.x) {
        float total = 0.0f;
        for (int w = 0; w < 8; ++w) total += warp_acc[w * E + e];
        partial[(int64_t)blockIdx.x * E + e] = total;
    }
}

// One warp per column: lane l adds chunks l, l + 32, ... in order, then a fixed shuffle tree adds the lanes.
// `partial2` (nullable): a second array with chunks2 rows, added after the first.
__global__ void __launch_bounds__(256) colsum_final_kernel(const float* __restrict__ partial, const float* __restrict__ partial2,
                                                           float* __restrict__ out, int chunks, int chunks2, int cols,
                                                           int accumulate) {
    grid_dependency_wait();
    grid_dependency_launch();
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= cols) return;
    float total = 0.0f;
    for (int i = lane; i < chunks; i += 32) total += partial[(int64_t)i * cols + c];
    if (partial2)
        for (int i = lane; i < chunks2; i += 32) total += partial2[(int64_t)i * cols + c];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) total += __shfl_xor_sync(0xffffffffu, total, off);
    if (lane == 0) out[c] = accumulate ? out[c] + total : total;
}

template <typename T>
__global__ void __launch_bounds__(256) splitk_reduce_kernel(const float* __restrict__ ws, int parts, int M, int N,
                                                            T* __restrict__ dst1, int m_split, T* __restrict__ dst2, int m2,
                                                            int accumulate) {
    grid_dependency_wait();
    grid_dependency_launch();
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;     // N is a multiple of 4
    if (i >= (int64_t)(m_split + m2) * N) return;
    const int m = (int)(i / N);
    float4 acc = *(const float4*)(ws + i);
    for (int s = 1; s < parts; ++s) {
        const float4 v = *(const float4*)(ws + (int64_t)s * M * N + i);
        acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
    T* dst = m < m_split ? dst1 + i : dst2 + (i - (int64_t)m_split * N);
    if (!(m < m_split ? dst1 : dst2)) return;
    if (accumulate) { acc.x += (float)dst[0]; acc.y += (float)dst[1]; acc.z += (float)dst[2]; acc.w += (float)dst[3]; }
    dst[0] = (T)acc.x; dst[1] = (T)acc.y; dst[2] = (T)acc.z; dst[3] = (T)acc.w;
}

// [x' | logits] from the fp32 partial results of a descend launch whose contraction was cut into parts (few tokens:
// the launch has too few output tiles to fill the SMs otherwise).  ws is [parts][T][r + E]; the first r columns of a
// row are added in part order and rounded to bf16 (x'), the other E stay fp32 (the gate logits).  r, E multiples of 4.
__global__ void __launch_bounds__(256) descend_reduce_kernel(const float* __restrict__ ws, int parts, int T, int r, int E,
                                                             __nv_bfloat16* __restrict__ x_lo, float* __restrict__ logits) {
    grid_dependency_wait();
    grid_dependency_launch();
    const int n = r + E;
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (i >= (int64_t)T * n) return;
    const int t = (int)(i / n), c = (int)(i - (int64_t)t * n);
    float4 acc = *(const float4*)(ws + i);
    for (int s = 1; s < parts; ++s) {
        const float4 v = *(const float4*)(ws + (int64_t)s * T * n + i);
        acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
    if (c < r) {
        __nv_bfloat162* dst = (__nv_bfloat162*)(x_lo + (int64_t)t * r + c);
        dst[0] = __floats2bfloat162_rn(acc.x, acc.y);
        dst[1] = __floats2bfloat162_rn(acc.z, acc.w);
    } else {
        *(float4*)(logits + (int64_t)t * E + (c - r)) = acc;
    }
}

// Per-expert column sums (expert-bias gradients), in two deterministic steps so that one long segment does not
// serialise.  Step 1, block (cg, e, s): slice s of kColsumSlices equal row ranges of expert e's padded segment; 32
// column-threads x 8 row-lanes, a thread adds rows lane, lane + 8, ... of its 16-byte column vector in order, then the
// 8 row-lanes are added in order -> partial[e][s][:].  Step 2 adds the slices in order.
template <typename T>
__global__ void __launch_bounds__(256) grouped_colsum_kernel(const uint4* __restrict__ src, const int32_t* __restrict__ poffsets,
                                                             float* __restrict__ partial, int vecs_per_row) {
    grid_dependency_wait();
    grid_dependency_launch();
    constexpr int V = Vec<T>::kElems;
    __shared__ float part[8][32 * V];
    const int e = blockIdx.y, slice = blockIdx.z, ct = threadIdx.x & 31, rl = threadIdx.x >> 5;
    const int c = blockIdx.x * 32 + ct;
    const int64_t r0 = poffsets[e], rows = poffsets[e + 1] - r0;
    const int64_t per = (rows + kColsumSlices - 1) / kColsumSlices;
    const int64_t first = r0 + slice * per, last = min(r0 + rows, first + per);
    float acc[V];
#pragma unroll
    for (int i = 0; i < V; ++i) acc[i] = 0.0f;
    if (c < vecs_per_row) {
        int64_t row = first + rl;
        for (; row + 24 < last; row += 32) {           // four rows in flight per thread
            uint4 q[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) q[u] = src[(row + 8 * u) * vecs_per_row + c];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float f[V];
                Vec<T>::unpack(q[u], f);
#pragma unroll
                for (int i = 0; i < V; ++i) acc[i] += f[i];
            }
        }
        for (; row < last; row += 8) {
            float f[V];
            Vec<T>::unpack(src[row * vecs_per_row + c], f);
#pragma unroll
            for (int i = 0; i < V; ++i) acc[i] += f[i];
        }
    }
#pragma unroll
    for (int i = 0; i < V; ++i) part[rl][ct * V + i] = acc[i];
    __syncthreads();
    const int width = vecs_per_row * V;
    for (int j = threadIdx.x; j < 32 * V; j += blockDim.x) {
        const int col = blockIdx.x * 32 * V + j;
        if (col >= width) continue;
        float total = 0.0f;
        for (int q = 0; q < 8; ++q) total += part[q][j];
        partial[((int64_t)e * kColsumSlices + slice) * width + col] = total;
    }
}
__global__ void __launch_bounds__(256) grouped_colsum_final_kernel(const float* __restrict__ partial, float* __restrict__ out,
                                                                   int64_t n, int width, int accumulate) {
    grid_dependency_wait();
    grid_dependency_launch();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;      // i = e * width + col
    if (i >= n) return;
    const int64_t e = i / width, col = i - e * width;
    float total = 0.0f;
    for (int s = 0; s < kColsumSlices; ++s) total += partial[(e * kColsumSlices + s) * width + col];
    out[i] = accumulate ? out[i] + total : total;
}

// The arrays one after another, each over the whole grid (the routing tables of a training call, handed to the caller:
// nine copies by the copy engine's path cost 4 us each, 36 us of 411 at 2999 tokens).
__global__ void __launch_bounds__(256) word_copies_kernel(const WordCopies c) {
    grid_dependency_wait();
    grid_dependency_launch();
    for (int a = 0; a < c.n; ++a)
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < c.words[a]; i += (int64_t)gridDim.x * blockDim.x)
            c.dst[a][i] = c.src[a][i];
}

inline int elem_bytes(int dtype) { return dtype == BIGMAC_BF16 ? 2 : 4; }
inline unsigned warp_blocks(int64_t warps) { return (unsigned)((warps + 7) / 8); }

}  // namespace

cudaError_t launch_dispatch(const void* src, void* grouped, const Tables& tb, int k, int width, int dtype,
                            int64_t max_prows, cudaStream_t stream) {
    if (max_prows == 0) return cudaSuccess;
    const int vecs = width * elem_bytes(dtype) / 16;
    return launch_chained(dispatch_kernel, warp_blocks((max_prows + kDispatchRows - 1) / kDispatchRows), 256, 0, stream, (const uint4*)src, (uint4*)grouped, tb.slot_of_prow,
                          tb.n_tiles, k, vecs, max_prows);
}

cudaError_t launch_combine(const void* grouped, void* dst, const float* w, const int32_t* prow_of_slot, int T, int k,
                           int width, int dtype, cudaStream_t stream, int dst_ld, bool may_drop) {
    if (T == 0) return cudaSuccess;
    const int vecs = width * elem_bytes(dtype) / 16;
    const int dvecs = (dst_ld ? dst_ld : width) * elem_bytes(dtype) / 16;
    const uint4* src = (const uint4*)grouped;
    uint4* out = (uint4*)dst;
    if (dtype == BIGMAC_BF16) {
        if (may_drop) return launch_chained(combine_kernel<__nv_bfloat16, true>, warp_blocks(T), 256, 0, stream, src, out, w, prow_of_slot, T, k, vecs, dvecs);
        return launch_chained(combine_kernel<__nv_bfloat16, false>, warp_blocks(T), 256, 0, stream, src, out, w, prow_of_slot, T, k, vecs, dvecs);
    } else {
        if (may_drop) return launch_chained(combine_kernel<float, true>, warp_blocks(T), 256, 0, stream, src, out, w, prow_of_slot, T, k, vecs, dvecs);
        return launch_chained(combine_kernel<float, false>, warp_blocks(T), 256, 0, stream, src, out, w, prow_of_slot, T, k, vecs, dvecs);
    }
    return cudaGetLastError();
}

cudaError_t launch_combine_parts(const void* parts, const MlpSlicing& sl, const int32_t* n_tiles, void* dst, const float* w,
                                 const int32_t* prow_of_slot, int T, int k, int width, cudaStream_t stream, bool may_drop) {
    if (T == 0) return cudaSuccess;
    const int quads = width / 4;
    const int64_t n = (int64_t)T * quads, stride = (int64_t)T * k * quads;
    const unsigned blocks = (unsigned)((n + 127) / 128);
    if (may_drop) return launch_chained(combine_parts_kernel<true>, blocks, 128, 0, stream, (const float4*)parts, n_tiles, sl, stride, (uint2*)dst, w, prow_of_slot, T, k, quads);
    return launch_chained(combine_parts_kernel<false>, blocks, 128, 0, stream, (const float4*)parts, n_tiles, sl, stride, (uint2*)dst, w, prow_of_slot, T, k, quads);
}

cudaError_t launch_combine_bwd(const void* dy_lo, const void* u, void* du, float* dp, const Tables& tb, void* dlogits, int T, int k,
                               int width, int E, int dl_width, int dl_ld, int dtype, cudaStream_t stream, bool chained) {
    if (T == 0) return cudaSuccess;
    const int vecs = width * elem_bytes(dtype) / 16;
    const unsigned blocks = warp_blocks(T) + E;
    auto launch = [&](auto kernel, auto* dl) {
        return launch_maybe_chained(chained, kernel, blocks, 256, 0, stream, (const uint4*)dy_lo, (const uint4*)u, (uint4*)du, dp, tb.prow_of_slot,
                                    tb.topk_w, tb.topk_idx, tb.counts, tb.poffsets, dl, T, k, vecs, E, dl_width, dl_ld);
    };
    if (dtype == BIGMAC_BF16)
        return k <= 2 ? launch(combine_bwd_kernel<__nv_bfloat16, 2, 2>, (__nv_bfloat16*)dlogits) : launch(combine_bwd_kernel<__nv_bfloat16, 8, 1>, (__nv_bfloat16*)dlogits);
    return k <= 2 ? launch(combine_bwd_kernel<float, 2, 2>, (float*)dlogits) : launch(combine_bwd_kernel<float, 8, 1>, (float*)dlogits);
}

cudaError_t launch_gate_bwd(float* dp, const Tables& tb, void* dlogits, int T, int E, int width, int ld, int k,
                            int dtype, cudaStream_t stream) {
    if (T == 0) return cudaSuccess;
    if (dtype == BIGMAC_BF16)
        (void)launch_chained(gate_bwd_kernel<__nv_bfloat16>, warp_blocks(T), 256, 0, stream, dp, tb.topk_w, tb.topk_idx,
                                                                          (__nv_bfloat16*)dlogits, T, E, width, ld, k);
    else
        (void)launch_chained(gate_bwd_kernel<float>, warp_blocks(T), 256, 0, stream, dp, tb.topk_w, tb.topk_idx, (float*)dlogits, T, E, width, ld, k);
    return cudaGetLastError();
}

cudaError_t launch_gate_colsum(const float* dl_slot, const Tables& tb, float* db, float* partial, int64_t N, int E,
                               bool accumulate, cudaStream_t stream, const float* aux_partial) {
    (void)launch_chained(colsum_slots_kernel, kColsumChunks, 256, sizeof(float) * 8 * E, stream, dl_slot, tb.topk_idx, partial, N, E);
    (void)launch_chained(colsum_final_kernel, (unsigned)((E + 7) / 8), 256, 0, stream, partial, aux_partial, db, kColsumChunks, kAuxChunks, E, accumulate);
    return cudaGetLastError();
}

cudaError_t launch_grouped_colsum(const void* src, const int32_t* poffsets, float* out, float* partial, int E, int width,
                                  int dtype, bool accumulate, cudaStream_t stream) {
    if (E == 0 || width == 0) return cudaSuccess;
    const int vecs = width * elem_bytes(dtype) / 16;
    dim3 grid((unsigned)((vecs + 31) / 32), (unsigned)E, (unsigned)kColsumSlices);
    if (dtype == BIGMAC_BF16)
        (void)launch_chained(grouped_colsum_kernel<__nv_bfloat16>, grid, 256, 0, stream, (const uint4*)src, poffsets, partial, vecs);
    else
        (void)launch_chained(grouped_colsum_kernel<float>, grid, 256, 0, stream, (const uint4*)src, poffsets, partial, vecs);
    const int64_t n = (int64_t)E * width;
    (void)launch_chained(grouped_colsum_final_kernel, (unsigned)((n + 255) / 256), 256, 0, stream, partial, out, n, width, accumulate ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_word_copies(const WordCopies& c, cudaStream_t stream) {
    int64_t most = 0;
    for (int a = 0; a < c.n; ++a) most = c.words[a] > most ? c.words[a] : most;
    if (most == 0) return cudaSuccess;
    const int64_t blocks = (most + 1023) / 1024;
    return launch_chained(word_copies_kernel, (unsigned)(blocks < 592 ? blocks : 592), 256, 0, stream, c);
}

cudaError_t launch_descend_reduce(const float* ws, int parts, int T, int r, int E, void* x_lo, float* logits,
                                  cudaStream_t stream) {
    const int64_t quads = (int64_t)T * (r + E) / 4;
    if (quads == 0) return cudaSuccess;
    return launch_chained(descend_reduce_kernel, (unsigned)((quads + 255) / 256), 256, 0, stream, ws, parts, T, r, E, (__nv_bfloat16*)x_lo, logits);
}

cudaError_t launch_splitk_reduce(const float* ws, int parts, int M, int N, void* dst1, int m_split, void* dst2, int m2,
                                 int dtype, bool accumulate, cudaStream_t stream) {
    const int64_t quads = (int64_t)(m_split + m2) * N / 4;
    if (quads == 0) return cudaSuccess;
    const unsigned blocks = (unsigned)((quads + 255) / 256);
    if (dtype == BIGMAC_BF16)
        (void)launch_chained(splitk_reduce_kernel<__nv_bfloat16>, blocks, 256, 0, stream, ws, parts, M, N, (__nv_bfloat16*)dst1, m_split,
                                                                      (__nv_bfloat16*)dst2, m2, accumulate);
    else
        (void)launch_chained(splitk_reduce_kernel<float>, blocks, 256, 0, stream, ws, parts, M, N, (float*)dst1, m_split, (float*)dst2, m2,
                                                               accumulate);
    return cudaGetLastError();
}

}  // namespace bigmac
