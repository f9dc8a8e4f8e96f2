// Which kernel runs the experts of a call, as far as sizes decide it.  Host code without a CUDA header, so that the rules run on the
// CPU too; the slicing is evaluated on the device as well.
#pragma once
#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define BIGMAC_HOST_DEVICE __host__ __device__
#else
#define BIGMAC_HOST_DEVICE
#endif

namespace bigmac {

constexpr int kPad = 128;          // expert segments are padded to multiples of this many rows internally

// ---- hidden width in slices, inference (gemm_tc_mlp.cu)
// How many slices is a function of the number of row tiles, which only the device knows: every kernel concerned
// evaluates mlp_slices for itself.
struct MlpSlicing {
    int units;       // SMs
    int chunks;      // 128-wide chunks of the hidden width
    int most;        // slices that the output buffer has room for
    int per_tile;    // work items per 128-row tile and slice
    unsigned long long inv;   // 2^40 / units, rounded up: division by a multiplication (exact below 2^40 / units^2)
};
// The slices s (a power of two) with the shortest longest SM: rounds of items, times an item's
// chunks and what its start and its output take in units of a chunk (fp32 partial results: twice the bytes of bf16).
// Few tiles: more slices put idle SMs to work (64 tiles of 8 chunks: two slices, 17 -> 12 us); more than one tile per SM:
// one slice (220 tiles of 8 chunks: the fp32 rows of two slices cost what the better last round gains; so does leaving the whole
// rounds uncut and cutting the rest only, 88 -> 90 us at 3001 tokens and no difference up to 13000).  The units were fitted at
// d 2048; against the best of 1, 2, 4 and 8 slices a forward of 24 to 4096 tokens is within 4.4 % at eight widths (r 64 to 512, h 256 to
// 2048, 8 to 128 experts), most within 1.5 %, but for d 4096 at 24 tokens (107.8 us, one slice 97.5).
// Slices that differ by a chunk, of at least three, are taken where one slice would leave half of the SMs idle (2 experts of
// h 2112, r 512, 64 tokens: 65 -> 41 us a forward, 32 experts 72 -> 60); with more tiles their fp32 rows cost more (100 experts, 600
// tokens: 106 -> 121), and slices of one or two chunks bring nothing at 500 tokens and more.
BIGMAC_HOST_DEVICE inline int mlp_slices(const MlpSlicing& m, int tiles) {
    int best = 1, best_cost = 0x7fffffff;
    for (int j = 0; (1 << j) <= m.most; ++j) {
        if ((m.chunks & ((1 << j) - 1)) && ((m.chunks >> j) < 3 || 2 * tiles > m.units)) break;
        const int rounds = (int)(((unsigned)(tiles * m.per_tile << j) + m.units - 1) * m.inv >> 40);
        const int cost = rounds * (((m.chunks - 1) >> j) + 1 + (j > 0 ? 3 : 2));
        if (cost < best_cost) { best = 1 << j; best_cost = cost; }
    }
    return best;
}
// Slices are limited to what fits the activation buffer [P, h] of bf16 that the separate contractions would use.
inline MlpSlicing mlp_slicing(int units, int r, int h, int64_t N, int64_t P) {
    MlpSlicing m{units, (h + 127) / 128, 1, r <= 256 ? 1 : 2, ((1ull << 40) + units - 1) / units};
    while (m.most < 8 && 2 * m.most * N * r * 4 <= P * h * 2) m.most *= 2;
    return m;
}

// ---- both contractions on CTA pairs (gemm_tc_ffn.cu)
// What the host knows of a call: N = T k rows over E experts, of which an expert keeps at most `cap`.
struct ExpertCall {
    int T, k, r, h, E, cap, units;         // units: SMs
    bool training;
    int64_t N() const { return (int64_t)T * k; }
};

// Rounds of pairs of 128-row tiles on the SM pairs: if the experts are chosen evenly, an expert has about N / E rows, give or take
// sqrt(N / E), and the probability that it reaches its j-th pair is taken as a ramp of two deviations to either side; if they
// are chosen as unevenly as Zipf's law has it, full pairs and 0.85 (few rows an expert) to 0.55 (2048) pairs an expert more, a fit within
// 2 % of the pairs to such loads of 32 and 64 experts.
inline double ffn_rounds(const ExpertCall& m, bool even) {
    const double N = (double)m.N(), pair = 2.0 * kPad, units = m.units / 2;
    if (!even) return (std::fmin(N, (double)m.cap * m.E) / pair + (0.5 + 0.42 / (1 + N / m.E / 300)) * m.E) / units;
    const double rows = std::fmin(N / m.E, (double)m.cap), dev = std::sqrt(N / m.E) + 1e-3;
    const int64_t whole = (int64_t)std::fmax(0.0, std::ceil((rows - 2 * dev) / pair));      // reached by all
    double pairs = (double)whole;
    for (int64_t j = whole; pair * j < rows + 2 * dev; ++j) pairs += std::fmin(1.0, 0.5 + (rows - pair * j) / (4 * dev));
    return pairs * m.E / units;
}

// Where the kernel on CTA pairs pays, among the widths it takes.
// Measured against the separate contractions, us (a training step; even loads; d 2048 r 256 h 1024 64 experts top-8, and d 1024 r 128
// h 512 32 experts top-4): it wins unless its last round of pairs is nearly empty.  How full that is depends on the loads, which only the
// device knows, so both estimates have to allow it.
//   r 256: 600 tokens 176 -> 172, 4000 288 -> 266, 12000 649 -> 640, Zipf 600 185 -> 179, 3000 286 -> 275, 16384 907 -> 874 (the SM clock rises
//          from 1.53 to 1.63 GHz under the power cap); 2048 (65 % of two rounds) 227 -> 229, Zipf 3500 (68 % of three) 303 -> 312.  1400: 207 ->
//          190 even, but Zipf (91 pairs for 64) 223 -> 232, and 850 Zipf (78) 196 -> 221
//   r 128: 300 103 -> 100, 3000 127 -> 121, 8000 178 -> 174, 20000 348 -> 339; but 4096 (1.1 rounds) 136 -> 146, 6000 (70 %) 159 -> 160,
//          9000 (72 %) 193 -> 197, 11000 (87 %) 215 -> 216; Zipf 3300 138 -> 132, 3600 142 -> 155
// Inference, against the kernel whose tokens are the N of its MMAs (gemm_tc_mlp.cu), which takes a batch's few rows an expert better:
//   r 256: 800 tokens (100 rows) 61 -> 63, 1200 (150) 64.8 -> 64.2, 3001 83 -> 77, 8000 145 -> 127, Zipf 1500 64 -> 75, 2300 (79 %) 80 -> 77, 3950 (73 %)
//   88 -> 95, 4200 (78 %) 100 -> 95;  r 128: 2000 (250) 37.1 -> 37.4, 2500 (312) 40.1 -> 40.1, 3500 41.2 -> 40.4, 4096 (1.1 rounds) 41.7 -> 46.2, 5000 (64 %)
//   54.2 -> 51.2, 12000 77 -> 70, Zipf 3300 40.9 -> 40.4, 3600 41 -> 47, 5000 53 -> 51.
// That kernel keeps u in fp32 where it cuts the hidden width (mlp_slices: up to half as many tiles as SMs, with more than ten chunks
// up to an eighth of the SMs for each chunk), which is more precise than u in bf16 here: a batch stays with it if its loads could
// leave so few tiles (under a capacity limit, if k experts are chosen by all tokens and keep what the limit allows).
inline bool ffn_pair_pays(const ExpertCall& m) {
    if (!m.training) {
        const double rows = std::fmin((double)m.N(), (double)m.cap * m.E), fewest = (double)m.k * std::fmin((double)m.T, (double)m.cap);
        const int chunks = m.h / 128;
        const double cut_up_to = 128.0 * m.units * (chunks <= 10 ? 0.5 : chunks / 8.0);        // rows
        if (fewest <= cut_up_to || rows < (m.r == 256 ? 150.0 : 320.0) * m.E) return false;
    }
    const double least = m.training ? (m.r == 256 ? 0.72 : 0.87) : (m.r == 256 ? 0.77 : 0.63);      // of all rounds' pairs
    for (int even = 0; even < 2; ++even) {
        const double rounds = ffn_rounds(m, even != 0), whole = std::ceil(1.03 * rounds);        // an estimate
        if (whole > 1 && rounds < least * whole) return false;
    }
    return true;
}

}  // namespace bigmac
