"""The rules that choose the experts' kernel from a call's sizes, on the CPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = r"""
#include <cstdio>
#include <initializer_list>
#include "expert_choice.h"
using namespace bigmac;
constexpr int kNoCapacity = 0x7fffffff;
static int capacity(double factor, int T, int k, int E) {
    const double N = (double)T * k, rows = factor > 0 ? std::ceil(factor * N / E) : N;
    return rows < N ? (int)rows : kNoCapacity;
}
"""


def _run(tmp_path, program, *args):
    src, exe = tmp_path / "choice.cpp", tmp_path / "choice"
    src.write_text(PRELUDE + program)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2502_16927_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    run = subprocess.run([str(exe), *map(str, args)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
    return run.stdout


def test_inference_on_pairs_only_where_u_was_in_bf16_anyway(tmp_path):
    """The kernel on CTA pairs rounds u to bf16.  The other one keeps it in fp32 where it cuts the hidden width, which it decides by the
    row tiles that the loads leave: no loads of a call that goes to the pairs may leave so few, also under a capacity limit."""
    out = _run(tmp_path, r"""
int main() {
    int chosen = 0, limited = 0;
    for (int r : {128, 256})
        for (int chunks : {1, 2, 3, 4, 7, 8, 10, 11, 12, 16, 24, 32, 64})
            for (int E : {1, 4, 8, 16, 33, 64, 128, 256})
                for (int k : {1, 2, 4, 8})
                    for (double factor : {0.0, 0.5, 1.0, 1.2, 2.0})
                        for (double t = 16; t < 40000; t *= 1.07) {
                            const int T = (int)t, h = 128 * chunks;
                            if (k > E) continue;
                            const int cap = capacity(factor, T, k, E);
                            if (!ffn_pair_pays(ExpertCall{T, k, r, h, E, cap, 148, false})) continue;
                            ++chosen;
                            limited += cap != kNoCapacity;
                            const int64_t N = (int64_t)T * k, P = ((N + 127) / 128 + E) * 128;
                            const MlpSlicing m = mlp_slicing(148, r, h, N, P);
                            // k experts take every token, as far as the limit lets them
                            const int64_t keep = T < cap ? T : cap;
                            for (int64_t tiles = k * ((keep + 127) / 128); tiles <= P / 128; ++tiles)
                                if (mlp_slices(m, (int)tiles) != 1) {
                                    std::printf("r %d h %d E %d k %d T %d capacity %g: %d tiles are cut\n", r, h, E, k, T, factor, (int)tiles);
                                    return 1;
                                }
                        }
    std::printf("%d %d\n", chosen, limited);
    return 0;
}
""")
    chosen, limited = map(int, out.split())
    assert chosen > 1000 and limited > 100


def test_pairs_only_where_they_were_the_faster_ones(tmp_path):
    """Calls on either side of the lines, each timed both ways (148 SMs; even and Zipf loads where the loads are not known): the ones that
    the kernel on CTA pairs made slower by 3 to 45 % keep their kernels, the ones that it made faster have it."""
    slower = [(1, 128, 512, 32, 4, 4200), (1, 128, 512, 32, 4, 1800), (1, 128, 1024, 8, 2, 300), (1, 128, 2048, 8, 2, 300), (1, 128, 2048, 8, 2, 3000),
              (1, 128, 4096, 8, 2, 32), (1, 128, 2048, 64, 2, 1678), (1, 128, 1024, 256, 8, 1280), (1, 128, 128, 256, 8, 9000), (1, 128, 512, 128, 2, 13177), (1, 256, 2048, 8, 2, 300),
              (1, 256, 2048, 8, 2, 3000), (1, 256, 2048, 64, 3, 286), (1, 256, 2048, 16, 1, 9386), (1, 256, 256, 256, 1, 3832), (1, 256, 256, 256, 8, 1000), (1, 256, 2048, 256, 8, 3000),
              (1, 256, 1024, 64, 8, 700), (1, 256, 1024, 64, 8, 20500), (1, 256, 1024, 256, 8, 32000), (0, 128, 2048, 128, 8, 6000),
              (0, 128, 1024, 64, 8, 4096), (0, 128, 512, 64, 8, 4096), (0, 128, 2048, 128, 8, 8192), (0, 128, 512, 32, 4, 8700), (0, 256, 1024, 128, 8, 3040),
              (0, 256, 2048, 128, 8, 6000), (0, 256, 1024, 64, 8, 1150), (0, 128, 128, 256, 8, 16384)]
    faster = [(1, 128, 512, 32, 4, 3000), (1, 128, 512, 32, 4, 16384), (1, 128, 2048, 8, 2, 8192), (1, 128, 256, 8, 2, 300),
              (1, 256, 1024, 64, 8, 2999), (1, 256, 1024, 64, 8, 5600), (1, 256, 1024, 64, 8, 16384), (1, 256, 256, 256, 8, 6080), (1, 256, 1024, 32, 4, 3000),
              (0, 128, 512, 32, 4, 5000), (0, 128, 512, 32, 4, 16384), (0, 256, 1024, 64, 8, 3001), (0, 256, 1024, 64, 8, 8000), (0, 256, 1024, 64, 8, 8700),
              (0, 256, 1024, 64, 8, 16384), (0, 256, 128, 64, 8, 3000)]
    shapes = slower + faster
    out = _run(tmp_path, r"""
#include <cstdlib>
int main(int argc, char** argv) {
    for (int i = 1; i + 5 < argc; i += 6) {
        int v[6];
        for (int j = 0; j < 6; ++j) v[j] = std::atoi(argv[i + j]);
        std::printf("%d\n", (int)ffn_pair_pays(ExpertCall{v[5], v[4], v[1], v[2], v[3], kNoCapacity, 148, v[0] != 0}));
    }
    return 0;
}
""", *(n for shape in shapes for n in shape))
    chosen = [s for s, c in zip(shapes, map(int, out.split())) if c]
    assert chosen == faster, (set(chosen) - set(faster), set(faster) - set(chosen))
