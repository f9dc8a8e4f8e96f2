// Both contractions of an expert in one launch of the fp32 path, for narrow experts (r <= 32, h <= 256):
//     forward   z = x W1_e^T, a = sigma(z), u = a W2_e^T       (training: a and sigma'(z) are written)
//     backward  dz = (du W2_e) sigma'(z), dxg = dz W1_e        (dz takes the place of sigma')
// At these widths a contraction is a chain of latencies (launch, table, operands, sum, store) around a microsecond of arithmetic:
// the second one now begins from shared memory where the first has left its output.
//
// A block has ROWS rows of one expert and walks the hidden width in chunks of 128 columns: both weight chunks and the rows are
// staged at once; a thread sums ROWS / 8 x 4 of the chunk's ROWS x 128 middle (its warp shares the rows: broadcasts; the columns are 32
// apart: no conflicts), then ROWS / 16 x r / 16 of the ROWS x r output, whose sums stay in registers over the chunks.  Four terms of the
// middle and sixteen of the output are added up before they join the others: the separate contractions, whose warps each have a
// part of the sum, are as exact; one running sum was 1.15 to 1.6 times as far from 64 bits (256 tokens 50.3 -> 50.6 us a training step).
// Bound by latency.  Blocks of 16 rows while four of them for an SM are enough, else of 32 (256 tokens, training: 59.5 us with 32
// rows, 58.4 with separate contractions, 55 with 16); blocks with nothing but padding rows only write the zeros that the weight
// gradients want there (55 -> 52).  Figures at uses_ffn_simt.
#include "act.cuh"
#include "internal.h"

namespace bigmac {

namespace {

constexpr int kChunk = 128, kThreads = 256, kMaxR = 32;
constexpr int LDC = kChunk + 4;                          // row length of what lies along the hidden width in shared memory

struct FfnSimtArgs {
    const float *x, *w1, *w2;                            // x: the rows (backward: du)
    float *mid, *sigma, *out;                            // mid: a (nullable: inference); sigma: sigma' out; backward: sigma' in, dz out
    int r, h, act, P;
    const int32_t *tile_expert, *n_tiles, *counts, *poffsets;
    int inv_qr;                                          // 2^16 / (r / 4), rounded up
};

// 16 bytes from global to shared memory; zeros where !there (the source is not read).
__device__ __forceinline__ void copy16(float* to, const float* from, bool there) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from), "r"(there ? 16u : 0u) : "memory");
}

template <bool BWD, int ROWS>
__global__ void __launch_bounds__(kThreads, 3) ffn_simt_kernel(const FfnSimtArgs p) {
    grid_dependency_wait();
    grid_dependency_launch();
    extern __shared__ float4 ffn_smem[];
    const int r = p.r, ldr = r + 4, tid = threadIdx.x;
    constexpr int RI = ROWS / 8, RO = ROWS / 16;         // rows of a thread in the middle and in the output
    const int row0 = blockIdx.x * ROWS, tile = row0 / kPad;
    if (tile >= *p.n_tiles) return;
    const int e = p.tile_expert[tile];
    if (row0 >= p.poffsets[e] + p.counts[e]) {           // padding rows alone: the weight gradients want zeros there
        float* mid = BWD ? p.sigma : p.mid;
        if (mid)
            for (int i = tid; i < ROWS * (p.h / 4); i += kThreads) reinterpret_cast<float4*>(mid + (int64_t)row0 * p.h)[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        return;
    }
    float* s_x = reinterpret_cast<float*>(ffn_smem);     // [ROWS][r + 4]
    float* s_w1 = s_x + ROWS * ldr;                     // [128][r + 4]
    float* s_w2 = s_w1 + kChunk * ldr;                   // [r][132]
    float* s_mid = s_w2 + r * LDC;                       // [ROWS][132]
    const float* w1 = p.w1 + (int64_t)e * p.h * r;
    const float* w2 = p.w2 + (int64_t)e * p.h * r;
    const int qr = r / 4;
    float out[RO][kMaxR / 16] = {};
    const int tm = tid >> 5, tn = tid & 31;              // the middle: rows RI tm + i, columns tn + 32 j
    const int om = RO * (tid >> 4), on = tid & 15;        // the output: rows om + i, columns on + 16 j
    for (int c0 = 0; c0 < p.h; c0 += kChunk) {
        const int width = min(kChunk, p.h - c0);         // a multiple of four
        __syncthreads();                                 // the chunk before is contracted
        // asynchronous copies: all of a thread's are in flight together
        if (c0 == 0)
            for (int i = tid; i < ROWS * qr; i += kThreads) {
                const int m = i * p.inv_qr >> 16, q = (i - m * qr) * 4;
                copy16(s_x + m * ldr + q, p.x + (int64_t)(row0 + m) * r + q, true);
            }
        for (int i = tid; i < kChunk * qr; i += kThreads) {
            const int n = i * p.inv_qr >> 16, q = (i - n * qr) * 4;
            copy16(s_w1 + n * ldr + q, w1 + (int64_t)(n < width ? c0 + n : 0) * r + q, n < width);
        }
        for (int i = tid; i < r * (kChunk / 4); i += kThreads) {
            const int c = i / (kChunk / 4), q = i % (kChunk / 4) * 4;
            copy16(s_w2 + c * LDC + q, w2 + (int64_t)c * p.h + (q < width ? c0 + q : 0), q < width);
        }
        float sig[RI][4];
        if (BWD) {                                       // sigma' is on its way beside the weights
#pragma unroll
            for (int i = 0; i < RI; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    sig[i][j] = tn + 32 * j < width ? p.sigma[(int64_t)(row0 + RI * tm + i) * p.h + c0 + tn + 32 * j] : 0.0f;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        float acc[RI][4] = {};
        for (int k = 0; k < r; k += 4) {
            float a[RI][4], b[4][4];                     // [row or column][k]
#pragma unroll
            for (int i = 0; i < RI; ++i) *reinterpret_cast<float4*>(a[i]) = *reinterpret_cast<const float4*>(s_x + (RI * tm + i) * ldr + k);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (!BWD) *reinterpret_cast<float4*>(b[j]) = *reinterpret_cast<const float4*>(s_w1 + (tn + 32 * j) * ldr + k);
                else
#pragma unroll
                    for (int q = 0; q < 4; ++q) b[j][q] = s_w2[(k + q) * LDC + tn + 32 * j];
            }
#pragma unroll
            for (int i = 0; i < RI; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)              // four terms, then to the others
                    acc[i][j] += fmaf(a[i][3], b[j][3], fmaf(a[i][2], b[j][2], fmaf(a[i][1], b[j][1], a[i][0] * b[j][0])));
        }
#pragma unroll
        for (int i = 0; i < RI; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) s_mid[(RI * tm + i) * LDC + tn + 32 * j] = BWD ? acc[i][j] * sig[i][j] : acc[i][j];
        // a thread's own, one copy of the activations' code (a copy of four of them for each element waited for instruction fetch)
#pragma unroll 1
        for (int q = 0; q < 4 * RI; ++q) {
            const int m = RI * tm + (q >> 2), n = tn + 32 * (q & 3);
            if (n >= width) continue;
            const int64_t at = (int64_t)(row0 + m) * p.h + c0 + n;
            float v = s_mid[m * LDC + n];
            if (BWD) p.sigma[at] = v;
            else {
                if (p.sigma) p.sigma[at] = act_grad(p.act, v);
                v = act_apply(p.act, v);
                s_mid[m * LDC + n] = v;
                if (p.mid) p.mid[at] = v;
            }
        }
        __syncthreads();
        for (int k0 = 0; k0 < width; k0 += 16) {         // sixteen terms, then to the others
            float part[RO][kMaxR / 16] = {};
#pragma unroll
            for (int kk = 0; kk < 16; kk += 4) {
                const int k = k0 + kk;
                if (k >= width) break;
                float a[RO][4];
#pragma unroll
                for (int i = 0; i < RO; ++i) *reinterpret_cast<float4*>(a[i]) = *reinterpret_cast<const float4*>(s_mid + (om + i) * LDC + k);
#pragma unroll
                for (int j = 0; j < kMaxR / 16; ++j) {
                    if (on + 16 * j >= r) continue;
                    float b[4];
                    if (!BWD) *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(s_w2 + (on + 16 * j) * LDC + k);
                    else
#pragma unroll
                        for (int q = 0; q < 4; ++q) b[q] = s_w1[(k + q) * ldr + on + 16 * j];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int i = 0; i < RO; ++i) part[i][j] = fmaf(a[i][q], b[q], part[i][j]);
                }
            }
#pragma unroll
            for (int i = 0; i < RO; ++i)
#pragma unroll
                for (int j = 0; j < kMaxR / 16; ++j) out[i][j] += part[i][j];
        }
    }
#pragma unroll
    for (int i = 0; i < RO; ++i)
#pragma unroll
        for (int j = 0; j < kMaxR / 16; ++j)
            if (on + 16 * j < r) p.out[(int64_t)(row0 + om + i) * r + on + 16 * j] = out[i][j];
}

template <bool BWD, int ROWS>
cudaError_t launch_rows(const FfnSimtArgs& p, cudaStream_t stream) {
    auto smem = [](int r) { return (int)sizeof(float) * ((ROWS + kChunk) * (r + 4) + r * LDC + ROWS * LDC); };
    static PerDeviceOnce once;
    int dev;
    if (once.needed(&dev)) {
        cudaError_t e = cudaFuncSetAttribute(ffn_simt_kernel<BWD, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem(kMaxR));
        if (e != cudaSuccess) return e;
        once.mark(dev);
    }
    return launch_chained(ffn_simt_kernel<BWD, ROWS>, (unsigned)(p.P / ROWS), kThreads, smem(p.r), stream, p);
}
template <bool BWD>
cudaError_t launch(const FfnSimtArgs& p, cudaStream_t stream) {
    if (p.P < kPad) return cudaSuccess;
    return p.P / 16 <= 4 * gemm_tc_sm_count() ? launch_rows<BWD, 16>(p, stream) : launch_rows<BWD, 32>(p, stream);
}

}  // namespace

bool ffn_simt_supported(int r, int h, int dtype) { return dtype == BIGMAC_F32 && r <= kMaxR && r % 4 == 0 && h <= 2 * kChunk && h % 4 == 0; }

cudaError_t launch_ffn_simt_forward(const void* xg, const void* w1, const void* w2, void* a, void* sigma, void* u, int64_t max_rows, int r, int h,
                                    int act, const Tables& tb, cudaStream_t stream) {
    return launch<false>(FfnSimtArgs{(const float*)xg, (const float*)w1, (const float*)w2, sigma ? (float*)a : nullptr, (float*)sigma, (float*)u, r, h, act,
                                     (int)max_rows, tb.tile_expert, tb.n_tiles, tb.counts, tb.poffsets, (65536 + r / 4 - 1) / (r / 4)}, stream);
}

cudaError_t launch_ffn_simt_backward(const void* du, const void* w1, const void* w2, void* sigma, void* dxg, int64_t max_rows, int r, int h,
                                     const Tables& tb, cudaStream_t stream) {
    return launch<true>(FfnSimtArgs{(const float*)du, (const float*)w1, (const float*)w2, nullptr, (float*)sigma, (float*)dxg, r, h, 0, (int)max_rows,
                                    tb.tile_expert, tb.n_tiles, tb.counts, tb.poffsets, (65536 + r / 4 - 1) / (r / 4)}, stream);
}

}  // namespace bigmac
