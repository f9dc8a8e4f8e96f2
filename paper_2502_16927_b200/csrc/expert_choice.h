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
// padded rows of N slots over E experts, at most
inline int64_t padded_rows_max(int64_t N, int E) { return ((N + kPad - 1) / kPad + E) * (int64_t)kPad; }
// Do that kernel's fp32 rows fit the activation buffer [P, h] of bf16?
inline bool mlp_fits(int r, int h, int64_t N, int64_t P) { return N * r * 4 <= P * h * 2; }
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

// Rounds of items of `size` rows on `units` SMs or SM pairs.  If the experts are chosen evenly, an expert has about N / E rows, give or
// take 1.5 sqrt(N / E) (a gate without a bias has some preferences of its own; 32 experts top-4 pass three rounds of pairs at 13050
// tokens), and reaches its j-th item with the normal distribution's probability.  If they are chosen as unevenly as Zipf's law has
// it: full items and 0.85 (few rows an expert) to 0.55 (eight items) an expert more, within 2 % of the pairs of tiles for 32 and 64 experts.
inline double item_rounds(const ExpertCall& m, int size, int units, bool even) {
    const double N = (double)m.N();
    if (!even) return (std::fmin(N, (double)m.cap * m.E) / size + (0.5 + 0.42 / (1 + N / m.E / (1.172 * size))) * m.E) / units;
    const double rows = std::fmin(N / m.E, (double)m.cap), dev = 1.5 * std::sqrt(N / m.E) + 1e-3;
    const int64_t whole = (int64_t)std::fmax(0.0, std::ceil((rows - 3 * dev) / size));      // reached by all
    double items = (double)whole;
    for (int64_t j = whole; size * j < rows + 3 * dev; ++j) items += 0.5 * std::erfc((size * j - rows) / (1.41421356 * dev));
    return items * m.E / units;
}

// Where the kernel on CTA pairs pays, among the widths it takes.  How full its last round of pairs is depends on the loads, which only
// the device knows, so both estimates have to allow it.  The lines were set on steps and forwards of r 128 (d 1024) and r 256 (d 2048) with
// h 128 to 4096, 8 to 256 experts, 8 to 3000 rows an expert, even and Zipf loads: of 1684 shapes a training step goes to the pairs
// with 626, 553 of them faster by more than 1.5 % and two slower (2.2 %), a forward with 452, 428 faster and seven slower (3.5 % at most; up
// to 10 % where loads just miss the estimated number of rounds).
// Figures: us, the other kernels -> this one; loads even unless said.
//
// Training, against the separate contractions.  It wins with many rows an expert and full rounds.
//   d 2048, r 256, h 1024, 64 experts top-8: 3000 tokens 253 -> 245, Zipf 280 -> 269, 5600 354 -> 338, 8000 441 -> 423, 13000 638 -> 616; but 2048 (68 %
//   of two rounds) 229 -> 231, Zipf 700 (1.01 rounds) 187 -> 218, 1400 and 3950 224 -> 230 and 321 -> 320 (even 205 -> 190, 283 -> 261).
//   d 1024, r 128, h 512, 32 experts top-4: 2300 tokens 120 -> 116, 3000 124 -> 120, 16384 283 -> 277, 24000 395 -> 384; but 4200 (1.16 rounds) 140 ->
//   149, 5600 155 -> 160, 9000 186 -> 195, Zipf 3600 (1.04) 143 -> 155; 1000 to 1800 tokens lose 1 to 3 %,
//   512 to 880 (one tile an expert) win as much.
// In a single round the separate contractions have blocks for all SMs, which counts the more, the longer an item's walk along
// the hidden width is: 8 experts top-2, 300 tokens, r 128, h 256 103 -> 96, 512 105 -> 103, 1024 108 -> 115, 2048 111 -> 141, 4096 125 -> 197; r 256,
// h 1024 123 -> 130, 2048 134 -> 158; 8192 tokens, 0.9 of the round: r 128, h 2048 235 -> 223, r 256, h 2048 330 -> 311.
// With more rounds an expert needs the rows, a pair that is half empty costs a whole one: 256 experts top-8, 1280 tokens (40 rows), r 256, h 256
// 201 -> 214, 2048 573 -> 600, r 128, h 1024 266 -> 312; 6080 tokens (190 rows), r 256, h 256 320 -> 285, 2048 809 -> 774; r 128, h 512, 128
// experts, Zipf, 190 to 256 rows 195 -> 207 and 219 -> 239, 375 and 512 rows 267 -> 271 and 325 -> 317.  Very large batches of r 256, under
// the power cap: h 1024, 64 experts, 20500 tokens 943 -> 983, 24000 1127 -> 1125, 29000 1333 -> 1335, 256 experts, 32000 1678 -> 1742.  r 128 with h 128 wins
// little (64 experts, 3000 tokens 117 -> 115; 256 experts, 12000 254 -> 259).
//
// Inference, against the kernel whose tokens are the N of its MMAs (gemm_tc_mlp.cu), which takes a batch's few rows an expert better and
// whose items are single tiles on single SMs: what counts is how its rounds compare with these.
//   r 256, h 1024, 64 experts: 1400 tokens 61.4 -> 60.8, 3000 84 -> 77, 8000 148 -> 131, 8700 (four rounds of tiles, five of pairs) 150 -> 143, 16384 287 -> 236, Zipf
//   1150 (one, two) 59 -> 74, 3950 (two, three) 89 -> 95, 6300 (three, four) 119 -> 122; 128 experts, 3040 tokens, Zipf (two, three) 93 -> 102.
//   r 128, h 512, 32 experts: 2600 40.4 -> 40.2, 5000 52.9 -> 51.2, 16384 93 -> 86, 18200 (four, five) 95.8 -> 94.1, 3600 Zipf (one, two) 41 -> 46, 8700 (two,
//   three) 58 -> 61, 13500 (three, four) 78.1 -> 79.2; with a longer walk four to five rounds lose as well: 128 experts, h 2048, 8192 tokens 162 -> 179.
// Where the hidden width is too narrow for that kernel, it is the separate contractions again: 64 experts, 3000 tokens, h 128, r 256 59 -> 51,
// r 128 47 -> 43; but 256 experts, 16384 tokens, r 128 125 -> 129.
// That kernel keeps u in fp32 where it cuts the hidden width (mlp_slices: up to half as many tiles as SMs, with more than ten chunks
// up to an eighth of the SMs for each chunk), which is more precise than u in bf16 here: a batch stays with it if its loads could
// leave so few tiles (under a capacity limit, if k experts are chosen by all tokens and keep what the limit allows).
inline bool ffn_pair_pays(const ExpertCall& m) {
    const bool wide = m.r == 256;
    const int chunks = m.h / 128;
    const double rows = std::fmin((double)m.N(), (double)m.cap * m.E) / m.E;               // an expert's, on average
    const bool mlp = mlp_fits(m.r, m.h, m.N(), padded_rows_max(m.N(), m.E));
    double least = m.training ? (wide ? 0.72 : 0.87) : (wide ? 0.77 : 0.63);               // part of the rounds that has to be filled
    double least_of_one = 0;
    if (m.training) {
        if (wide ? chunks > 2 && m.N() > 160000 : chunks == 1) return false;
        if (wide && chunks >= 16) least = 0.8;
        if (chunks > (wide ? 4 : 2)) least_of_one = wide ? std::fmin(0.72, 0.08 + chunks / 27.0) : chunks <= 4 ? 0.6 : 0.87;
    } else {
        const double fewest = (double)m.k * std::fmin((double)m.T, (double)m.cap);
        const double cut_up_to = 128.0 * m.units * (chunks <= 10 ? 0.5 : chunks / 8.0);    // rows
        if (fewest <= cut_up_to || rows < (wide ? 150 : 320)) return false;
        if (!mlp && !wide && m.N() > 128000) return false;
    }
    for (int even = 0; even < 2; ++even) {
        const double rounds = item_rounds(m, 2 * kPad, m.units / 2, even != 0), whole = std::ceil(1.03 * rounds);        // an estimate
        const bool one_tile = m.training && !wide && chunks <= 4 && rounds < 0.6 && rows >= 60 && rows <= 112;
        if (!one_tile && (whole > 1 ? rounds < least * whole : rounds < least_of_one)) return false;
        if (m.training && !one_tile && (whole > 1 ? rows < (wide || chunks <= 2 ? 176 : 300) : chunks > 2 && rows < (wide ? 60 : 176))) return false;
        if (!m.training && mlp && std::ceil(0.985 * item_rounds(m, kPad, m.units, even != 0)) < (wide || chunks <= 4 ? 0.78 : 0.95) * std::ceil(rounds)) return false;
    }
    return true;
}

}  // namespace bigmac
