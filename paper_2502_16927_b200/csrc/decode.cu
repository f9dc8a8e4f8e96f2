// Small-batch (decode-shaped) inference forward of the BigMac layer in ONE cooperative kernel.
//
// For a handful of tokens the layer is a chain of matrix-vector products that is bound by streaming the touched weights
// once (W'_down, W_gate, the selected experts' W1/W2, W'_up) and by latency; separate launches cost far more than the
// arithmetic.  All SMs walk five phases:
//   A  [x' | logits] = x [W'_down ; W_gate]^T   a CTA owns a few weight rows, a warp takes 32 16-byte pieces of one
//   B  top-k + softmax gate values               a warp per token, repeated by every CTA in its own shared memory
//   C  a = sigma(W1_e x') per routed slot         a CTA owns a range of hidden units, a warp takes a few rows
//   D  y' = sum_j p_j W2_{e_j} a_j                a CTA owns some columns of one token, a warp takes (column, slot) rows
//   E  y = W'_up y'                               a CTA owns a few rows
// Values that cross from one CTA to another (x', logits, a, y') travel as 8-byte words (fp32 value, tag of this launch):
// the consumer polls the very words it needs until their tags match, so a hand-over is one store and one load through
// L2.  With a grid-wide barrier (arrive, spin, then load) each of the three hand-overs took 2.2-2.7 us, 7 of the 15 us of
// one token.  The words are written by this kernel only, in memory that one handle at a time has and that was zero at first;
// the tag counts the launches on that memory, on the device (a captured launch can be replayed).  A tag has 32 bits and would
// meet itself after 2^32 launches (17 hours of one-token calls): so every launch also retags one word a block of those that its
// own batch does not use, in turn, and no word is ever older than a few thousand launches.  A stale word never matches.
// Code is executed once or a few times per launch, and a first execution waits for instruction fetch: phases are small
// loops, ranges and divisors come ready from the host.  (Four extra warps that ran through the later phases' code
// beforehand, without effect, gained nothing: what is left is the latency of the hand-overs and of the weights.)
// Weights do not depend on the hand-overs: W'_up rows are fetched into shared memory at the start, the first rows of A
// before x is staged, the first W2 rows before the wait for a; C fetches a step's rows ahead.
// Products accumulate in fp32, intermediates stay fp32.  The cooperative launch guarantees that all CTAs run at the same
// time; every wait is bounded (status word), so the kernel always ends.
#include "internal.h"
#include "act.cuh"

namespace bigmac {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kDecodeThreads = 512, kWarps = kDecodeThreads / 32;
constexpr int kDecodeMaxTokens = 16;        // 16 tokens: 18.6 us against 26 of the launch chain at d 1024, 33.0 against 35.7 at d 2048
constexpr int kDecodeMaxExperts = 256;
constexpr int kDecodeMaxSlots = 2048;       // T k: every CTA keeps all slots' expert ids and gate values
// Hidden activations of one token staged in shared memory at a time (128 KB).  (64 KB, two passes for k h = 32768: 2 tokens of d 2048,
// r 256, h 4096, 64 experts, k 8 24.4 -> 27.8 us.)
constexpr int kDecodeMaxHidden = 32768;
constexpr int kDecodeMaxUpBytes = 65536;    // W'_up rows of a CTA kept in shared memory (56 KB at d 8192, r 512: 4 tokens 24.0 -> 22.6 us)
constexpr size_t kDecodeMaxWords = 1u << 20; // hand-over words (8 MB) a handle keeps at most

// n / d for 0 <= n < 2^31 by a multiplication (d >= 1; round-up method with a 31-bit dividend).
struct Divisor {
    uint32_t d, m, s;
    Divisor() = default;
    explicit Divisor(int v) : d((uint32_t)v), m(0), s(0) {
        while (s < 31 && (1u << s) < d) ++s;
        m = (uint32_t)(((1ull << (31 + s)) + d - 1) / d);
    }
    __device__ __forceinline__ int div(int n) const { return (int)(uint32_t)(((unsigned long long)(uint32_t)n * m) >> (31 + s)); }
};
// Share b of `total` things dealt out over the grid in contiguous ranges.
struct Split {
    int per, rest;
    Split() = default;
    Split(int total, int grid) : per(total / grid), rest(total % grid) {}
    __device__ __forceinline__ int first(int b) const { return b * per + min(b, rest); }
};

struct DecodeArgs {
    const __nv_bfloat16 *x, *w_gate, *w_down, *w1, *w2, *w_up;
    const float* b_gate;
    __nv_bfloat16* y;
    unsigned long long *x_lo, *logits, *a, *y_lo;      // hand-over words: [T,r], [T,LE], [T*k,h], [T,r]
    int32_t* topk_idx;
    float* topk_w;
    unsigned* epoch;                   // [grid] launches on this memory so far, a word of its own for every CTA
    int used, total;                   // hand-over words of this launch, and of the memory that x_lo begins
    unsigned sweep;                    // launches in which every word has its turn to be retagged, less one (a power of two, less one)
    int* status;
    int T, d, r, h, E, k, act;
    int copies, copy_words;            // x', logits and y' are written `copies` times, copy_words apart; CTA b reads copy b % copies
    int LE;                            // row length of the logits' words: E up to a multiple of four
    Split rows_a, groups_c, rows_e;    // who does what in phases A, C (groups of rows of all slots) and E
    Split cols_d;                      // phase D: columns of a token over its CTAs
    int ctas_d;                        // phase D: CTAs per token
    Divisor by_parts, by_pieces, by_k, by_slot, by_ctas, by_pass;   // parts of a row in A; pieces of x; k; groups of a slot in C; ctas_d; slots of a pass in D
    // shared memory, offsets in floats: region (x; then x'; then a of a token; then y'), W'_up rows, logits, slots, sums
    int up_rows, off_up, off_log, off_idx, off_w, off_sums;
};
extern __shared__ float4 decode_smem_raw[];
__device__ __forceinline__ float* smem_at(int off) { return reinterpret_cast<float*>(decode_smem_raw) + off; }

__device__ __forceinline__ void unpack8(const uint4& v, float* f) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        f[2 * i] = __uint_as_float(w[i] << 16);
        f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}

// ---- hand-over words.  Value and tag share one 64-bit access, so neither needs an ordering with anything else.
__device__ __forceinline__ void put_word(unsigned long long* p, float v, uint32_t tag) {
    const unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ void put_copies(const DecodeArgs& a, unsigned long long* p, float v, uint32_t tag) {
#pragma unroll 1
    for (int i = 0; i < a.copies; ++i) put_word(p + i * a.copy_words, v, tag);
}
// Thread `tid` of `threads` waits for its share of n words (n even, 16-byte aligned) and puts the values into dst, in the
// words' own order.  A thread asks for four pairs at a time, and only for its own: a pair that everybody reads holds all of
// them up.
__device__ __noinline__ void get_words(float* dst, const unsigned long long* words, int n, int tid, int threads, uint32_t tag, int* status) {
    constexpr int U = 4;
#pragma unroll 1
    for (int i0 = 2 * tid; i0 < n; i0 += 2 * U * threads) {
        unsigned long long w[2 * U];
        bool ok = false;
#pragma unroll 1
        for (uint32_t spin = 0; spin < (1u << 20) && !ok; ++spin) {
            ok = true;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + 2 * u * threads < n)
                    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w[2 * u]), "=l"(w[2 * u + 1]) : "l"(words + i0 + 2 * u * threads) : "memory");
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + 2 * u * threads < n) ok = ok && (uint32_t)(w[2 * u] >> 32) == tag && (uint32_t)(w[2 * u + 1] >> 32) == tag;
        }
        if (!ok) atomicExch(status, 1);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + 2 * u * threads < n)
                *reinterpret_cast<float2*>(dst + i0 + 2 * u * threads) = make_float2(__uint_as_float((uint32_t)w[2 * u]), __uint_as_float((uint32_t)w[2 * u + 1]));
    }
}

// Where element e of a staged vector of n elements (a multiple of 8) sits: elements 8c .. 8c+3 at float4 number c,
// elements 8c+4 .. 8c+7 at float4 number n / 8 + c.  Neighbouring lanes, which hold neighbouring 16-byte pieces of a
// bf16 row, then read neighbouring 16 bytes of shared memory, where the natural layout has a two-way bank conflict.
__device__ __forceinline__ int split_index(int e, int n) { return ((e >> 2) & 1) * (n >> 1) + ((e >> 3) << 2) + (e & 3); }

// Dot product of one 16-byte piece of a bf16 row (unpacked to four pairs) with elements 8c .. 8c+7 of a vector staged as
// above (v0, v1), added to a pair of partial sums: packed multiply-adds, two elements an instruction.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) { f32x2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) { f32x2 d; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c)); return d; }
__device__ __forceinline__ float sum2(f32x2 v) { float a, b; asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); return a + b; }
struct Piece {
    f32x2 w[4];
    __device__ __forceinline__ explicit Piece(const uint4& v) {
        float f[8];
        unpack8(v, f);
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = pack2(f[2 * i], f[2 * i + 1]);
    }
};
__device__ __forceinline__ f32x2 dot8(const Piece& q, const float4& v0, const float4& v1, f32x2 acc) {
    acc = fma2(q.w[0], pack2(v0.x, v0.y), acc);
    acc = fma2(q.w[1], pack2(v0.z, v0.w), acc);
    acc = fma2(q.w[2], pack2(v1.x, v1.y), acc);
    return fma2(q.w[3], pack2(v1.z, v1.w), acc);
}

// Sums each of the N values (a power of two, at most 32) over the warp's lanes with N - 1 + log2(32 / N) shuffles
// instead of 5 N: every halving step a lane hands half of its values to its partner and keeps the sums of the
// other half.  Returns the total of value number lane / (32 / N); v is used up.  The order of the additions is fixed.
template <int N>
__device__ __forceinline__ float warp_reduce_scatter(float* v) {
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int cnt = N; cnt > 1; cnt >>= 1, off >>= 1) {
        const bool upper = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < cnt / 2; ++i) {
            const float send = upper ? v[i] : v[i + cnt / 2];
            const float keep = upper ? v[i + cnt / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(kFull, send, off);
        }
    }
    float total = v[0];
#pragma unroll
    for (int o = 16 / N; o > 0; o >>= 1) total += __shfl_xor_sync(kFull, total, o);
    return total;
}

// A: the rows of [W'_down ; W_gate] of this CTA (the gate reads x, not x'); a warp takes 32 pieces of one row at a time, the
// parts of a row meet in shared memory and are added in order.  TG: tokens whose sums a warp keeps at a time.
template <int TG>
__device__ __forceinline__ void phase_a(const DecodeArgs& p, uint32_t tag) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x;
    float* xs = smem_at(0);
    float* sums = smem_at(p.off_sums);
    const int pieces = p.d / 8, parts = (int)p.by_parts.d, r0 = p.rows_a.first(b), nrows = p.rows_a.first(b + 1) - r0, tasks = nrows * parts;
    auto fetch = [&](int i) {
        const int row = p.by_parts.div(i), c = (i - row * parts) * 32 + lane, j = r0 + row;
        const uint4* w = reinterpret_cast<const uint4*>(j < p.r ? p.w_down : p.w_gate) + (int64_t)(j < p.r ? j : j - p.r) * pieces;
        return c < pieces ? __ldg(w + c) : make_uint4(0u, 0u, 0u, 0u);
    };
    uint4 wv = make_uint4(0u, 0u, 0u, 0u);
    if (warp < tasks) wv = fetch(warp);                      // on its way before x
    constexpr int XU = TG == 1 ? 1 : 4;
    const int xn = p.T * pieces;
#pragma unroll 1
    for (int i0 = tid; i0 < xn; i0 += XU * kDecodeThreads) {
        uint4 xv[XU];
#pragma unroll
        for (int u = 0; u < XU; ++u)
            if (i0 + u * kDecodeThreads < xn) xv[u] = __ldg(reinterpret_cast<const uint4*>(p.x) + i0 + u * kDecodeThreads);
#pragma unroll
        for (int u = 0; u < XU; ++u)
            if (i0 + u * kDecodeThreads < xn) {
                float f[8];
                unpack8(xv[u], f);
                const int t = p.by_pieces.div(i0 + u * kDecodeThreads), q = i0 + u * kDecodeThreads - t * pieces;
                float4* vt = reinterpret_cast<float4*>(xs + t * p.d);
                vt[q] = make_float4(f[0], f[1], f[2], f[3]);
                vt[pieces + q] = make_float4(f[4], f[5], f[6], f[7]);
            }
    }
    if (p.up_rows > 0) {                                     // W'_up for phase E
        const int up0 = p.rows_e.first(b), n = (p.rows_e.first(b + 1) - up0) * (p.r / 8);
        const uint4* from = reinterpret_cast<const uint4*>(p.w_up) + (int64_t)up0 * (p.r / 8);
        const uint32_t to = (uint32_t)__cvta_generic_to_shared(smem_at(p.off_up));
#pragma unroll 1
        for (int i = tid; i < n; i += kDecodeThreads)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + i * 16), "l"(from + i) : "memory");
    }
    __syncthreads();
#pragma unroll 1
    for (int i = warp; i < tasks; i += kWarps) {
        const Piece q(wv);
        const int c = min((i - p.by_parts.div(i) * parts) * 32 + lane, pieces - 1);   // lanes past the end hold zero weights
        if (i + kWarps < tasks) wv = fetch(i + kWarps);
#pragma unroll 1
        for (int t0 = 0; t0 < p.T; t0 += TG) {
            float acc[TG];
#pragma unroll
            for (int t = 0; t < TG; ++t) {
                const float4* vt = reinterpret_cast<const float4*>(xs + min(t0 + t, p.T - 1) * p.d);
                acc[t] = sum2(dot8(q, vt[c], vt[pieces + c], 0ull));
            }
            const float sum = warp_reduce_scatter<TG>(acc);          // token t0 + lane / (32 / TG)
            if (!(lane & (32 / TG - 1))) sums[i * 16 + t0 + lane / (32 / TG)] = sum;   // tokens past T: slots of their own
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < nrows * 16; i += kDecodeThreads) {
        const int t = i & 15, j = r0 + (i >> 4), e = j - p.r;
        if (t >= p.T) continue;
        float sum = 0.0f;
#pragma unroll 4
        for (int q = 0; q < parts; ++q) sum += sums[((i >> 4) * parts + q) * 16 + t];
        unsigned long long* to = p.x_lo + t * p.r + split_index(j, p.r);
        if (e >= 0) {
            if (p.b_gate) sum += p.b_gate[e];
            sum = sum == sum ? sum : -INFINITY;              // NaN is ordered as -inf
            to = p.logits + t * p.LE + e;
            if (e == p.E - 1)                                // words that fill the row up: never counted before anything
#pragma unroll 1
                for (int q = p.E; q < p.LE; ++q) put_copies(p, p.logits + t * p.LE + q, __int_as_float(0x7fffffff), tag);
        }
        put_copies(p, to, sum, tag);
    }
}

// Floats as unsigned integers of the same order (both zeros alike).
__device__ __forceinline__ uint32_t order_key(float v) {
    const uint32_t b = __float_as_uint(v + 0.0f);
    return b ^ (uint32_t)((int32_t)b >> 31 | (int32_t)0x80000000);
}

// The experts of one token by one warp: rounds of arg-max over the lanes' experts lane + 32 q (E <= 32 Q), in registers.  (Counting
// the experts before each expert takes no rounds, but E^2 T comparisons: 35.1 us instead of 33.5 for 16 tokens of 64 experts, 59
// instead of 17 for 16 of 256 at d 1024, r 128, h 512, k 2.)
template <int Q>
__device__ __forceinline__ void select_experts(const float* l, int* idx, int E, int k) {
    const int lane = threadIdx.x & 31;
    uint32_t key[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) key[q] = lane + 32 * q < E ? max(order_key(l[lane + 32 * q]), 1u) : 0u;
#pragma unroll 1
    for (int j = 0; j < k; ++j) {
        uint32_t mine = key[0];
#pragma unroll
        for (int q = 1; q < Q; ++q) mine = max(mine, key[q]);
        const uint32_t best = __reduce_max_sync(kFull, mine);
        uint32_t e = kDecodeMaxExperts;
#pragma unroll
        for (int q = Q - 1; q >= 0; --q) e = key[q] == best ? lane + 32 * q : e;
        e = __reduce_min_sync(kFull, e);
#pragma unroll
        for (int q = 0; q < Q; ++q) key[q] = lane + 32 * q == e ? 0u : key[q];
        if (lane == 0) idx[j] = (int)e;
    }
}

// B: top-k by (logit descending, expert id ascending), softmax over the k kept logits; x' takes x's place.
__device__ __forceinline__ void phase_b(const DecodeArgs& p, uint32_t tag) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int half = kDecodeThreads / 2;
    const bool logits = tid < half;
    float* s_log = smem_at(p.off_log);
    int* s_idx = reinterpret_cast<int*>(smem_at(p.off_idx));
    float* s_w = smem_at(p.off_w);
    __syncthreads();
    get_words(smem_at(logits ? p.off_log : 0), (logits ? p.logits : p.x_lo) + blockIdx.x % p.copies * p.copy_words, logits ? p.T * p.LE : p.T * p.r, tid & (half - 1), half, tag, p.status);
    __syncthreads();
    // a warp per token (T <= 16 warps)
    if (warp < p.T) {
        if (p.E <= 64) select_experts<2>(s_log + warp * p.LE, s_idx + warp * p.k, p.E, p.k);
        else select_experts<kDecodeMaxExperts / 32>(s_log + warp * p.LE, s_idx + warp * p.k, p.E, p.k);
    }
    __syncthreads();
    if (warp < p.T) {
        const int at = warp * p.k;
        const float* l = s_log + warp * p.LE;
        const float top = l[s_idx[at]];
        float sum = 0.0f;
#pragma unroll 1
        for (int j = lane; j < p.k; j += 32) {
            const float ex = top == -INFINITY ? 1.0f : expf(l[s_idx[at + j]] - top);      // only -inf logits kept: 1/k each
            s_w[at + j] = ex;
            sum += ex;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
#pragma unroll 1
        for (int j = lane; j < p.k; j += 32) {
            const float w = s_w[at + j] / sum;
            s_w[at + j] = w;
            if (blockIdx.x == 0) { p.topk_idx[at + j] = s_idx[at + j]; p.topk_w[at + j] = w; }
        }
    }
}

// C: a = sigma(W1_e x') per routed slot, ROWS rows per warp and step.  (Grouping the slots by expert, so that a weight byte
// is read once however many tokens chose the expert, was measured slower at every T <= 16: the repeats are L2 hits, and
// the lists and wider reductions cost more than they save.)
template <int ROWS>
__device__ __forceinline__ void phase_c(const DecodeArgs& p, uint32_t tag) {
    const int lane = threadIdx.x & 31, b = blockIdx.x, rp = p.r / 8;
    const int* s_idx = reinterpret_cast<const int*>(smem_at(p.off_idx));
    const int per_slot = (int)p.by_slot.d, g1 = p.groups_c.first(b + 1);     // h is a multiple of 16
    int g = p.groups_c.first(b) + (int)(threadIdx.x >> 5);
    uint4 wv[ROWS];
    const uint4* w = nullptr;
    auto rows_at = [&](int q) {
        const int s = p.by_slot.div(q);
        w = reinterpret_cast<const uint4*>(p.w1) + ((int64_t)s_idx[s] * p.h + (q - s * per_slot) * ROWS) * rp;
    };
    auto fetch = [&](int c) {
#pragma unroll
        for (int i = 0; i < ROWS; ++i) wv[i] = c < rp ? __ldg(w + i * rp + c) : make_uint4(0u, 0u, 0u, 0u);
    };
    if (g < g1) { rows_at(g); fetch(lane); }
#pragma unroll 1
    for (; g < g1; g += kWarps) {
        const int s = p.by_slot.div(g), q0 = (g - s * per_slot) * ROWS;
        const float4* v = reinterpret_cast<const float4*>(smem_at(p.by_k.div(s) * p.r));
        f32x2 acc2[ROWS] = {};
#pragma unroll 1
        for (int c = lane; c - lane < rp; c += 32) {
            const int cc = min(c, rp - 1);                   // lanes past the end hold zero weights
            const float4 v0 = v[cc], v1 = v[rp + cc];
#pragma unroll
            for (int i = 0; i < ROWS; ++i) acc2[i] = dot8(Piece(wv[i]), v0, v1, acc2[i]);
            int next = c + 32;                               // the next pieces, or the next step's rows, before the sums are finished
            if (next - lane >= rp && g + kWarps < g1) { rows_at(g + kWarps); next = lane; }
            fetch(next);
        }
        float acc[ROWS];
#pragma unroll
        for (int i = 0; i < ROWS; ++i) acc[i] = sum2(acc2[i]);
        constexpr int L = 32 / ROWS;
        const float z = act_apply(p.act, warp_reduce_scatter<ROWS>(acc));              // row lane / L
        if (!(lane & (L - 1))) put_word(p.a + (int64_t)s * p.h + split_index(q0 + lane / L, p.h), z, tag);
    }
}

// D: y'[t, c] = sum_j p_j (W2_{e_j}[c, :] a_j): floor(grid / T) CTAs per token, some columns each, ROWS (column, slot) rows per
// warp and step; in passes over groups of slots where a token's hidden activations are more than shared memory takes.
// MANY: more passes than one.
template <int ROWS, bool MANY>
__device__ __forceinline__ void phase_d(const DecodeArgs& p, uint32_t tag) {
    const int tid = threadIdx.x, lane = tid & 31, b = blockIdx.x, hp = p.h / 8;
    const int* s_idx = reinterpret_cast<const int*>(smem_at(p.off_idx));
    const float* s_w = smem_at(p.off_w);
    float* sums = smem_at(p.off_sums);
    const bool works = b < p.T * p.ctas_d;           // the last grid - T floor(grid / T) CTAs have no columns: rows = 0
    const int t = works ? p.by_ctas.div(b) : 0, share = works ? b - t * p.ctas_d : 0, c0 = p.cols_d.first(share);
    const int per_pass = MANY ? (int)p.by_pass.d : p.k;      // slots of a pass
    const int rows = works ? (p.cols_d.first(share + 1) - c0) * per_pass : 0;    // row i of a pass: column c0 + i / per_pass, slot i % per_pass
    const int* experts = s_idx + t * p.k;
    uint4 wv[ROWS][4];
    const uint4* w[ROWS];
    int slot[ROWS];
    int left = p.k;                                          // slots of this pass and those after it
    auto rows_at = [&](int i) {                              // rows i, i + kWarps, ...
#pragma unroll
        for (int n = 0; n < ROWS; ++n) {
            const int row = min(i + n * kWarps, max(rows - 1, 0)), col = p.by_pass.div(row);
            slot[n] = row - col * per_pass;
            if (MANY) slot[n] = min(slot[n], left - 1);      // (the last pass may have fewer slots: rows that count for nothing)
            w[n] = reinterpret_cast<const uint4*>(p.w2) + ((int64_t)experts[slot[n]] * p.r + c0 + col) * hp;
        }
    };
    auto fetch = [&](int c) {                                // four pieces of a lane
#pragma unroll
        for (int n = 0; n < ROWS; ++n)
#pragma unroll
            for (int u = 0; u < 4; ++u) wv[n][u] = c + 32 * u < hp ? __ldg(w[n] + c + 32 * u) : make_uint4(0u, 0u, 0u, 0u);
    };
    const unsigned long long* words = p.a + (int64_t)t * p.k * p.h;
    const float4* v = reinterpret_cast<const float4*>(smem_at(0));
#pragma unroll 1
    for (float* pass = sums; left > 0; pass += rows, experts += per_pass, words += per_pass * p.h, left = MANY ? left - per_pass : 0) {
        int i = tid >> 5;
        rows_at(i);
        if (i < rows) fetch(lane);                           // the first rows are on their way before the wait for a
        __syncthreads();                                     // x' or the slots before are not read any more, their place takes a
        if (rows > 0) get_words(smem_at(0), words, (MANY ? min(per_pass, left) : p.k) * p.h, tid, kDecodeThreads, tag, p.status);
        __syncthreads();
#pragma unroll 1
        for (; i < rows; i += ROWS * kWarps) {
            f32x2 acc2[ROWS] = {};
            int from[ROWS];
#pragma unroll
            for (int n = 0; n < ROWS; ++n) from[n] = 2 * slot[n] * hp;
#pragma unroll 1
            for (int c = lane; c - lane < hp; c += 128) {
#pragma unroll
                for (int n = 0; n < ROWS; ++n)
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int at = from[n] + min(c + 32 * u, hp - 1);        // past the end: zero weights
                        acc2[n] = dot8(Piece(wv[n][u]), v[at], v[at + hp], acc2[n]);
                    }
                int next = c + 128;
                if (next - lane >= hp && i + ROWS * kWarps < rows) { rows_at(i + ROWS * kWarps); next = lane; }
                fetch(next);
            }
            float acc[ROWS];
#pragma unroll
            for (int n = 0; n < ROWS; ++n) acc[n] = sum2(acc2[n]);
            constexpr int L = 32 / ROWS;
            const float u = warp_reduce_scatter<ROWS>(acc);                      // row lane / L
            const int row = i + lane / L * kWarps;
            if (!(lane & (L - 1)) && row < rows) pass[row] = u;
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int c = tid; c * per_pass < rows; c += kDecodeThreads) {  // combine in slot order
        float acc = 0.0f;
        const float* from = sums + c * per_pass;
#pragma unroll 1
        for (int j0 = 0; j0 < (MANY ? p.k : 1); j0 += per_pass, from += rows)
#pragma unroll 4
            for (int j = 0; j < (MANY ? min(per_pass, p.k - j0) : p.k); ++j) acc = fmaf(s_w[t * p.k + j0 + j], from[j], acc);
        put_copies(p, p.y_lo + t * p.r + split_index(c0 + c, p.r), acc, tag);
    }
}

// E: ascend, one row of W'_up per warp and step (a is not read any more: the barrier before the combine of D).
template <int TG>
__device__ __forceinline__ void phase_e(const DecodeArgs& p, uint32_t tag) {
    const int tid = threadIdx.x, lane = tid & 31, b = blockIdx.x, rp = p.r / 8;
    get_words(smem_at(0), p.y_lo + b % p.copies * p.copy_words, p.T * p.r, tid, kDecodeThreads, tag, p.status);
    asm volatile("cp.async.wait_all;" ::: "memory");     // the rows of W'_up
    __syncthreads();
    const int up0 = p.rows_e.first(b), up1 = p.rows_e.first(b + 1);
#pragma unroll 1
    for (int row = up0 + (tid >> 5); row < up1; row += kWarps) {
        const uint4* w = p.up_rows > 0 ? reinterpret_cast<const uint4*>(smem_at(p.off_up)) + (row - up0) * rp : reinterpret_cast<const uint4*>(p.w_up) + (int64_t)row * rp;
#pragma unroll 1
        for (int t0 = 0; t0 < p.T; t0 += TG) {
            f32x2 acc2[TG] = {};
#pragma unroll 1
            for (int c = lane; c < rp; c += 32) {
                const Piece q(w[c]);
#pragma unroll
                for (int t = 0; t < TG; ++t) {
                    const float4* v = reinterpret_cast<const float4*>(smem_at(min(t0 + t, p.T - 1) * p.r));
                    acc2[t] = dot8(q, v[c], v[rp + c], acc2[t]);
                }
            }
            float acc[TG];
#pragma unroll
            for (int t = 0; t < TG; ++t) acc[t] = sum2(acc2[t]);
            constexpr int L = 32 / TG;
            const float sum = warp_reduce_scatter<TG>(acc);                  // token t0 + lane / L
            if (!(lane & (L - 1)) && t0 + lane / L < p.T) p.y[(int64_t)(t0 + lane / L) * p.d + row] = __float2bfloat16(sum);
        }
    }
}

// TG 1: for one or two tokens, where every phase is a single chain of latencies; TG 4: four tokens' sums at a time, more
// loads in flight per warp.  Three tokens: 16.8 us by TG 4, 17.1 by TG 1 at d 2048, 30.9 and 35.7 at d 4096.  Two tokens: 15.2 and
// 15.1 at d 2048 (k h = 8192), but 25.5 and 27.2 at d 4096 (k h = 16384), 20.6 and 21.1 at d 8192.
template <int TG, bool MANY>
__global__ void __launch_bounds__(kDecodeThreads, 1) decode_forward_kernel(const __grid_constant__ DecodeArgs p) {
    constexpr int ROWS_C = TG == 1 ? 4 : 8, ROWS_D = TG == 1 ? 1 : 2;
    uint32_t tag;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(tag) : "l"(p.epoch + blockIdx.x) : "memory");
    ++tag;
    phase_a<TG>(p, tag);
    if (threadIdx.x == kDecodeThreads - 1) {                 // (while the logits are on their way)
        const int i = (int)((tag & p.sweep) * gridDim.x + blockIdx.x);
        if (i >= p.used && i < p.total) put_word(p.x_lo + i, 0.0f, tag);
    }
    phase_b(p, tag);
    phase_c<ROWS_C>(p, tag);
    phase_d<ROWS_D, MANY>(p, tag);
    phase_e<TG>(p, tag);
    if (threadIdx.x == 0) p.epoch[blockIdx.x] = tag;         // nobody else reads or writes this CTA's word
}

constexpr size_t kDecodeSmemLimit = 220 * 1024;

// Shared memory of a launch, offsets in floats: the region that x, x', a and y' take in turn, rows of
// W'_up, and the rest.
size_t decode_smem(DecodeArgs& p, int grid) {
    const int T = p.T, d = p.d, r = p.r, h = p.h, E = p.E, k = p.k;
    int region = T * (d > r ? d : r);
    const int passes = (k * h + kDecodeMaxHidden - 1) / kDecodeMaxHidden, per_pass = (k + passes - 1) / passes;     // phase D
    if (per_pass * h > region) region = per_pass * h;
    p.by_pass = Divisor(per_pass);
    const int up = (d + grid - 1) / grid;
    p.LE = (E + 3) / 4 * 4;
    p.up_rows = 0;
    const int per_token = grid / T > 1 ? grid / T : 1, rows = ((r + per_token - 1) / per_token) * passes * per_pass;     // phase D's rows of a CTA
    const int sums_a = ((r + E + grid - 1) / grid) * ((d / 8 + 31) / 32) * 16, sums = rows > sums_a ? rows : sums_a;   // phase A's parts
    const size_t rest = (size_t)((region + 3) / 4 * 4) + T * p.LE + 2 * T * k + sums;
    if ((size_t)up * r * 2 <= kDecodeMaxUpBytes && sizeof(float) * rest + (size_t)up * r * 2 <= kDecodeSmemLimit) p.up_rows = up;
    p.off_up = (region + 3) / 4 * 4;
    p.off_log = p.off_up + p.up_rows * r / 2;                // r is a multiple of 8
    p.off_idx = p.off_log + T * p.LE;
    p.off_w = p.off_idx + T * k;
    p.off_sums = p.off_w + T * k;
    return sizeof(float) * ((size_t)p.off_sums + sums);
}
// Where x', logits and y' are a few lines of memory that all CTAs poll, copies keep the readers from queueing up (14.2 -> 13.9 us
// for one token, 19.4 -> 18.7 for four at r = 256; nothing for eight).
constexpr int decode_copies(int T, int r) { return T * r <= 512 ? 4 : T * r <= 1024 ? 2 : 1; }

DecodeArgs decode_shape(int T, int d, int r, int h, int E, int k) {
    DecodeArgs p{};
    p.T = T; p.d = d; p.r = r; p.h = h; p.E = E; p.k = k;
    return p;
}

}  // namespace

// Every slot streams its expert's weights for itself, from L2 where another had them before; the launch chain reads them once.
// From more than two slots an expert and 48 million weights a matrix streamed on the chain is the faster one (d 2048, r 512, h 2048, 64
// experts, k 16: 8 tokens 79.6 us against 81.2, 12 tokens 110 against 82; d 1024, r 256, h 8192, 16 experts, k 6: 4 tokens 45.4
// against 52.1, 6 tokens 57.9 against 53.0), with fewer weights it is not (r 128, h 512, 64 experts, k 32: 8 tokens 30.8 against 36.5).
static bool streams_too_much(int T, int r, int h, int E, int k) { return (int64_t)T * k > 2 * E && (int64_t)T * k * h * r > 48000000; }

bool decode_forward_supported(int T, int d, int r, int h, int E, int k, int dtype, int num_sms) {
    if (dtype != BIGMAC_BF16 || T < 1 || T > kDecodeMaxTokens || (int64_t)T * d > 32768 || d % 8 || r % 8 || h % 16 ||
        E > kDecodeMaxExperts || h > kDecodeMaxHidden || T * k > kDecodeMaxSlots || streams_too_much(T, r, h, E, k) || T > num_sms ||
        decode_forward_words(T, r, h, E, k) > kDecodeMaxWords)
        return false;
    DecodeArgs p = decode_shape(T, d, r, h, E, k);
    return decode_smem(p, num_sms) <= kDecodeSmemLimit;
}

// Hand-over words of batches of up to T tokens.
size_t decode_forward_words(int T, int r, int h, int E, int k) {
    size_t most = 0;
    for (int t = 1; t <= T; ++t) {
        const size_t words = (size_t)t * (decode_copies(t, r) * (2 * (size_t)r + (E + 3) / 4 * 4) + (size_t)k * h);
        if (words > most) most = words;
    }
    return most;
}

// The largest batch of at most max_tokens tokens that the kernel takes at these widths (0: none).
int decode_forward_max_tokens(int max_tokens, int d, int r, int h, int E, int k, int dtype, int num_sms) {
    int T = max_tokens < kDecodeMaxTokens ? max_tokens : kDecodeMaxTokens;
    while (T > 0 && !decode_forward_supported(T, d, r, h, E, k, dtype, num_sms)) --T;
    return T;
}

cudaError_t launch_decode_forward(const void* x, const bigmac_weights_t* W, void* y, void* words, size_t word_count, int32_t* topk_idx,
                                  float* topk_w, unsigned* epoch, int* status, int T, int d, int r, int h, int E, int k, int act,
                                  int num_sms, cudaStream_t stream) {
    DecodeArgs p = decode_shape(T, d, r, h, E, k);
    const size_t smem = decode_smem(p, num_sms);
    p.x = (const __nv_bfloat16*)x; p.w_gate = (const __nv_bfloat16*)W->w_gate; p.w_down = (const __nv_bfloat16*)W->w_down;
    p.w1 = (const __nv_bfloat16*)W->w1; p.w2 = (const __nv_bfloat16*)W->w2; p.w_up = (const __nv_bfloat16*)W->w_up;
    p.b_gate = W->b_gate; p.y = (__nv_bfloat16*)y;
    p.copies = decode_copies(T, r);
    p.copy_words = T * (2 * r + p.LE);
    p.x_lo = (unsigned long long*)words;
    p.logits = p.x_lo + (size_t)T * r;
    p.y_lo = p.logits + (size_t)T * p.LE;
    p.a = p.x_lo + (size_t)p.copies * p.copy_words;
    p.used = p.copies * p.copy_words + T * k * h;
    p.total = (int)word_count;
    if ((size_t)p.used > word_count || word_count > kDecodeMaxWords) return cudaErrorInvalidValue;
    while ((size_t)(p.sweep + 1) * num_sms < word_count) p.sweep = 2 * p.sweep + 1;
    p.topk_idx = topk_idx; p.topk_w = topk_w; p.epoch = epoch; p.status = status; p.act = act;
    const bool few = T == 1 || (T == 2 && k * h <= 8192 && d <= 4096);
    const int rows_c = few ? 4 : 8;
    p.rows_a = Split(r + E, num_sms); p.rows_e = Split(d, num_sms); p.groups_c = Split(T * k * (h / rows_c), num_sms);
    p.ctas_d = num_sms / T > 1 ? num_sms / T : 1; p.cols_d = Split(r, p.ctas_d);
    p.by_parts = Divisor((d / 8 + 31) / 32); p.by_pieces = Divisor(d / 8); p.by_k = Divisor(k); p.by_slot = Divisor(h / rows_c);
    p.by_ctas = Divisor(p.ctas_d);
    static PerDeviceOnce once;
    int dev;
    const void* kernels[2][2] = {{(const void*)decode_forward_kernel<4, false>, (const void*)decode_forward_kernel<4, true>},
                                 {(const void*)decode_forward_kernel<1, false>, (const void*)decode_forward_kernel<1, true>}};
    if (once.needed(&dev)) {
        for (int i = 0; i < 4; ++i) {
            const cudaError_t e = cudaFuncSetAttribute(kernels[i / 2][i % 2], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecodeSmemLimit);
            if (e != cudaSuccess) return e;
        }
        once.mark(dev);
    }
    void* ptrs[] = {(void*)&p};
    return cudaLaunchCooperativeKernel(kernels[few][(int)p.by_pass.d < k], dim3(num_sms), dim3(kDecodeThreads), ptrs, smem, stream);
}

}  // namespace bigmac
