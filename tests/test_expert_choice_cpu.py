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
