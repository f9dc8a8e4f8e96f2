// Plain FMA GEMM: C[m,n] (+)= epilogue(sum_k A(m,k) B(n,k)), fp32 accumulation in a fixed order.
// This is the arithmetic of the fp32 layer (tensor cores have no true-fp32 mode, and the routing margin and the 1e-4
// tolerance of that path need one) and a debugging reference for the bf16 path.
//
// The fp32 layer is used at small sizes, where every contraction is one short chain of latencies: one kernel runs up to
// five independent contractions (a launch costs more than most of them), a block stages a long k slice of its tile at
// once, its eight warps share the slice (each sums its own part of the k range into a 32 x 32 tile, 4 x 8 outputs per
// lane), and where the contraction is long a cluster of blocks shares it, the partial tiles meeting in distributed shared
// memory.  All sums have a fixed order.  Tiles: 32 x 32 with 128-deep slices (eight warps along k) while that many tiles do
// not fill the SMs twice, else 64 x 64 with 64-deep slices (2 x 2 warps, two along k: half the operand traffic).
// A training step of d 128, r 32, h 128, 8 experts, with one 64 x 64 tile kernel of 16-deep slices (a global round trip and
// two barriers per slice) and a launch per contraction before: 209 -> 62 us at 256 tokens, 800 -> 107 at 2048.
#include "tc_pair.cuh"
#include "act.cuh"

namespace bigmac {

namespace {

using tc::cluster_sync_all;
using tc::map_to_cta;

constexpr int kThreads = 256;

struct SimtBatch {
    GemmArgs g[kSimtBatch];
    int first[kSimtBatch + 1];     // first block of each problem
    int split[kSimtBatch];         // blocks (of one cluster) that share the contraction: 1 or the cluster size
};

template <typename T> struct Load4;
template <> struct Load4<float> {
    static __device__ __forceinline__ float4 vec(const float* p) { return *reinterpret_cast<const float4*>(p); }
};
template <> struct Load4<__nv_bfloat16> {
    static __device__ __forceinline__ float4 vec(const __nv_bfloat16* p) {
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
    }
};

// Four consecutive elements of row `row`, from column `col` on; zeros outside [0, rows) x [0, cols).
template <typename T>
__device__ __forceinline__ float4 load4(const T* base, int64_t ld, int row, int col, int rows, int cols, bool vec) {
    if (row >= rows || col >= cols) return make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const T* p = base + (int64_t)row * ld + col;
    if (vec && col + 4 <= cols) return Load4<T>::vec(p);
    float4 v = make_float4((float)p[0], 0.0f, 0.0f, 0.0f);
    if (col + 1 < cols) v.y = (float)p[1];
    if (col + 2 < cols) v.z = (float)p[2];
    if (col + 3 < cols) v.w = (float)p[3];
    return v;
}

// One output tile.  WK warps along k, (8 / WK) over the tile; TS = tile side, KC = k slice.
template <typename T, bool A_K, bool B_K, int WK>
__device__ __forceinline__ void simt_tile(const GemmArgs& g, int split, int tile_index, float* smem) {
    constexpr int TS = WK == 8 ? 32 : 64, KC = WK == 8 ? 128 : 64, WS = TS / 32;
    // operand in shared memory: as it lies in global memory, [row][k] or [k][row], 4 floats of padding per row
    constexpr int LDK = KC + 4, LDM = TS + 4;
    constexpr int OPERAND = TS * LDK > KC * LDM ? TS * LDK : KC * LDM;
    constexpr int NV = TS * KC / 4 / kThreads;               // vectors of an operand per thread and slice
    float* As = smem;
    float* Bs = smem + OPERAND;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tiles_n = (g.N + TS - 1) / TS, tiles_m = (g.M + TS - 1) / TS;
    const int e = g.group == GROUP_K ? tile_index / (tiles_m * tiles_n) : 0;
    const int r = tile_index - e * tiles_m * tiles_n, m0 = r / tiles_n * TS, n0 = r % tiles_n * TS;
    const T* A = (const T*)g.A;
    const T* B = (const T*)g.B;
    const float* bias = nullptr;
    int m_limit = g.M, k_begin = 0, k_end = g.K;
    int64_t c_base = 0;
    bool live = true;
    if (g.group == GROUP_M) {
        const int tile = m0 / kPad;
        live = tile < *g.n_tiles;                            // the same for all blocks of a cluster that shares a tile
        if (live) {
            const int expert = g.tile_expert[tile];
            B += (int64_t)expert * g.b_stride;
            if (g.bias) bias = g.bias + (int64_t)expert * g.bias_stride;
            m_limit = min(g.M, *g.n_tiles * kPad);
        }
    } else if (g.group == GROUP_K) {
        k_begin = g.poffsets[e];
        k_end = g.poffsets[e + 1];
        c_base = (int64_t)e * g.c_stride;
    }
    if (!live) return;                                       // (a shared tile is never of this kind: see the launch)
    const int rank = split > 1 ? (int)tc::cluster_ctarank() : 0;
    if (split > 1) {                                         // whole slices per block
        const int per = ((k_end - k_begin + split - 1) / split + KC - 1) / KC * KC;
        k_begin = min(k_begin + rank * per, k_end);
        k_end = min(k_begin + per, k_end);
    }
    const bool vec_a = g.lda % 4 == 0 && (uintptr_t)A % (4 * sizeof(T)) == 0, vec_b = g.ldb % 4 == 0 && (uintptr_t)B % (4 * sizeof(T)) == 0;
    const bool vec_b2 = g.ldb2 % 4 == 0 && (uintptr_t)g.B2 % (4 * sizeof(T)) == 0;
    const int b_end = g.B2 ? min(k_end, g.b2_first_k) : k_end;       // k rows of the first (MN-major) B tensor

    float4 va[NV], vb[NV];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int v = tid + i * kThreads;
            if (A_K) va[i] = load4(A, g.lda, m0 + v / (KC / 4), k0 + v % (KC / 4) * 4, m_limit, k_end, vec_a);
            else va[i] = load4(A, g.lda, k0 + v / (TS / 4), m0 + v % (TS / 4) * 4, k_end, m_limit, vec_a);
            if (B_K) vb[i] = load4(B, g.ldb, n0 + v / (KC / 4), k0 + v % (KC / 4) * 4, g.N, k_end, vec_b);
            else {
                const int k = k0 + v / (TS / 4), n = n0 + v % (TS / 4) * 4;
                vb[i] = g.B2 && k >= g.b2_first_k ? load4((const T*)g.B2, g.ldb2, k - g.b2_first_k, n, k_end - g.b2_first_k, g.N, vec_b2)
                                                  : load4(B, g.ldb, k, n, b_end, g.N, vec_b);
            }
        }
    };
    const int wk = warp / (WS * WS), wm = warp / WS % WS, wn = warp % WS;    // WS = 1: wm = wn = 0
    const int tm = lane >> 2, tn = lane & 3;
    // K-major operand: a lane's rows are tm + 8 i and columns tn + 4 j; MN-major: 4 tm + i and 4 tn + 16 (j / 4) + j % 4
    const float* a_from = A_K ? As + (wm * 32 + tm) * LDK : As + wm * 32 + 4 * tm;
    const float* b_from = B_K ? Bs + (wn * 32 + tn) * LDK : Bs + wn * 32 + 4 * tn;
    float acc[4][8] = {};
    if (k_begin < k_end) fetch(k_begin);
    for (int k0 = k_begin; k0 < k_end; k0 += KC) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int v = tid + i * kThreads;
            *reinterpret_cast<float4*>(A_K ? As + v / (KC / 4) * LDK + v % (KC / 4) * 4 : As + v / (TS / 4) * LDM + v % (TS / 4) * 4) = va[i];
            *reinterpret_cast<float4*>(B_K ? Bs + v / (KC / 4) * LDK + v % (KC / 4) * 4 : Bs + v / (TS / 4) * LDM + v % (TS / 4) * 4) = vb[i];
        }
        __syncthreads();
        if (k0 + KC < k_end) fetch(k0 + KC);
        const int ka = wk * (KC / WK), kb = min(ka + KC / WK, (k_end - k0 + 3) / 4 * 4);     // past the end: zeros
#pragma unroll 2
        for (int k = ka; k < kb; k += 4) {
            float a[4][4], b[8][4];                          // [row][k]
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 v = *reinterpret_cast<const float4*>(A_K ? a_from + 8 * i * LDK + k : a_from + (k + i) * LDM);
                if (A_K) { a[i][0] = v.x; a[i][1] = v.y; a[i][2] = v.z; a[i][3] = v.w; }
                else { a[0][i] = v.x; a[1][i] = v.y; a[2][i] = v.z; a[3][i] = v.w; }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float4 v = *reinterpret_cast<const float4*>(B_K ? b_from + 4 * j * LDK + k : b_from + (k + j / 2) * LDM + 16 * (j & 1));
                if (B_K) { b[j][0] = v.x; b[j][1] = v.y; b[j][2] = v.z; b[j][3] = v.w; }
                else { const int n = 4 * (j & 1), q = j / 2; b[n][q] = v.x; b[n + 1][q] = v.y; b[n + 2][q] = v.z; b[n + 3][q] = v.w; }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i][q], b[j][q], acc[i][j]);
        }
    }
    // ---- the warps' partial tiles, then the blocks', in order
    constexpr int LDR = 36;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int m = A_K ? tm + 8 * i : 4 * tm + i, n = B_K ? tn + 4 * j : 4 * tn + 16 * (j / 4) + j % 4;
            smem[(warp * 32 + m) * LDR + n] = acc[i][j];
        }
    __syncthreads();
    constexpr int Q = TS * TS / 4 / kThreads;                // groups of four outputs per thread
    float4 out[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int o = tid + q * kThreads, m = o / (TS / 4), n = o % (TS / 4) * 4;
        const int w0 = WS == 1 ? 0 : (m / 32) * WS + n / 32;
        float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int w = 0; w < WK; ++w) {
            const float4 v = *reinterpret_cast<const float4*>(smem + ((w * WS * WS + w0) * 32 + m % 32) * LDR + n % 32);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        out[q] = s;
    }
    int first = 0, last = TS * TS / 4;                       // output groups this block stores
    if (split > 1) {
        float4* whole = reinterpret_cast<float4*>(smem + 8 * 32 * LDR);      // behind the warps' tiles
#pragma unroll
        for (int q = 0; q < Q; ++q) whole[tid + q * kThreads] = out[q];
        cluster_sync_all();
        const int per = TS * TS / 4 / split;                 // split is a power of two
        first = rank * per;
        last = first + per;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int o = tid + q * kThreads;
            if (o < first || o >= last) continue;
            float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            for (int p = 0; p < split; ++p) {
                float4 v;
                asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(map_to_cta(whole + o, p)));
                s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
            }
            out[q] = s;
        }
    }
    const bool wide = g.ldc % 4 == 0 && (uintptr_t)g.C % 16 == 0 && c_base % 4 == 0;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int o = tid + q * kThreads, gm = m0 + o / (TS / 4), gn = n0 + o % (TS / 4) * 4;
        if (o < first || o >= last || gm >= m_limit || gn >= g.N) continue;
        const int64_t off = c_base + (int64_t)gm * g.ldc + gn;
        float v[4] = {out[q].x, out[q].y, out[q].z, out[q].w};
        const int count = min(4, g.N - gn);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= count) break;
            if (bias) v[j] += bias[gn + j];
            if (g.epilogue == EPI_ACT) {
                if (g.Z) ((T*)g.Z)[off + j] = (T)act_grad(g.act, v[j]);
                v[j] = act_apply(g.act, v[j]);
            } else if (g.epilogue == EPI_DACT) {
                v[j] *= (float)((const T*)g.Z)[off + j];
            }
        }
        if ((sizeof(T) == 4 || g.out_f32) && wide && count == 4) {
            float4* C = reinterpret_cast<float4*>((float*)g.C + off);
            if (g.accumulate) { const float4 c = *C; v[0] += c.x; v[1] += c.y; v[2] += c.z; v[3] += c.w; }
            *C = make_float4(v[0], v[1], v[2], v[3]);
            continue;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= count) break;
            if (g.out_f32) {
                float* C = (float*)g.C + off + j;
                *C = g.accumulate ? *C + v[j] : v[j];
            } else {
                T* C = (T*)g.C + off + j;
                *C = (T)(g.accumulate ? (float)*C + v[j] : v[j]);
            }
        }
    }
    if (split > 1) cluster_sync_all();                       // nobody leaves while others read its tile
}

template <typename T, int WK>
__global__ void __launch_bounds__(kThreads) gemm_simt_kernel(const __grid_constant__ SimtBatch batch) {
    grid_dependency_wait();
    grid_dependency_launch();
    extern __shared__ float4 simt_smem[];
    float* smem = reinterpret_cast<float*>(simt_smem);
    const int b = blockIdx.x;
    int i = 0;
    while (i + 1 < kSimtBatch && b >= batch.first[i + 1]) ++i;
    const GemmArgs& g = batch.g[i];
    const int split = batch.split[i], tile = (b - batch.first[i]) / split;
    const int TS = WK == 8 ? 32 : 64;
    if (tile >= ((g.M + TS - 1) / TS) * ((g.N + TS - 1) / TS) * (g.group == GROUP_K ? g.num_experts : 1)) return;   // fills a cluster
    if (g.a_kmajor) {
        if (g.b_kmajor) simt_tile<T, true, true, WK>(g, split, tile, smem);
        else simt_tile<T, true, false, WK>(g, split, tile, smem);
    } else {
        if (g.b_kmajor) simt_tile<T, false, true, WK>(g, split, tile, smem);
        else simt_tile<T, false, false, WK>(g, split, tile, smem);
    }
}

template <typename T, int WK>
cudaError_t launch(const GemmArgs* g, int count, cudaStream_t stream) {
    constexpr int TS = WK == 8 ? 32 : 64, KC = WK == 8 ? 128 : 64;
    SimtBatch b{};
    // A contraction of more than four slices is shared by four blocks, of more than eight by eight.  Not a row-grouped one,
    // whose dead tiles leave early, nor one per expert, whose lengths only the device knows.
    int cluster = 1;
    for (int i = 0; i < count; ++i)
        if (g[i].group == GROUP_NONE) {
            const int want = g[i].K > 8 * KC ? 8 : g[i].K > 4 * KC ? 4 : 1;
            if (want > cluster) cluster = want;
        }
    int64_t blocks = 0;
    for (int i = 0; i < kSimtBatch; ++i) {
        b.first[i] = (int)blocks;
        b.split[i] = 1;
        if (i >= count || g[i].M <= 0 || g[i].N <= 0) continue;
        b.g[i] = g[i];
        if (g[i].group == GROUP_NONE && g[i].K > 2 * KC) b.split[i] = cluster;
        const int64_t tiles = (int64_t)((g[i].M + TS - 1) / TS) * ((g[i].N + TS - 1) / TS) * (g[i].group == GROUP_K ? g[i].num_experts : 1);
        blocks += (tiles * b.split[i] + cluster - 1) / cluster * cluster;
    }
    b.first[kSimtBatch] = (int)blocks;
    if (blocks == 0) return cudaSuccess;
    if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
    constexpr int LDK = KC + 4, LDM = TS + 4, OPERAND = TS * LDK > KC * LDM ? TS * LDK : KC * LDM;
    constexpr size_t tiles_bytes = (8 * 32 * 36 + TS * TS) * sizeof(float), op_bytes = 2 * OPERAND * sizeof(float);
    constexpr size_t smem = tiles_bytes > op_bytes ? tiles_bytes : op_bytes;
    static PerDeviceOnce once;
    int dev;
    if (once.needed(&dev)) {
        cudaError_t e = cudaFuncSetAttribute(gemm_simt_kernel<T, WK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        once.mark(dev);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (switches().chain) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster; attr[n].val.clusterDim.y = 1; attr[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = attr; cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, gemm_simt_kernel<T, WK>, b);
}

}  // namespace

cudaError_t gemm_simt_batch(const GemmArgs* g, int count, int dtype, cudaStream_t stream) {
    if (count > kSimtBatch) return cudaErrorInvalidValue;
    int64_t wide = 0;                                        // 64 x 64 tiles
    for (int i = 0; i < count; ++i) {
        if (g[i].M <= 0 || g[i].N <= 0) continue;
        wide += (int64_t)((g[i].M + 63) / 64) * ((g[i].N + 63) / 64) * (g[i].group == GROUP_K ? g[i].num_experts : 1);
    }
    const bool small = wide < 2 * (int64_t)gemm_tc_sm_count();
    if (dtype == BIGMAC_BF16) return small ? launch<__nv_bfloat16, 8>(g, count, stream) : launch<__nv_bfloat16, 2>(g, count, stream);
    return small ? launch<float, 8>(g, count, stream) : launch<float, 2>(g, count, stream);
}

cudaError_t gemm_simt(const GemmArgs& g, int dtype, cudaStream_t stream) { return gemm_simt_batch(&g, 1, dtype, stream); }

}  // namespace bigmac
