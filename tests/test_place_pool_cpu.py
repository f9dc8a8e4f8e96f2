"""The pool of static device memory for small-batch handles, on the CPU with a fake of the device calls: a place is given back
only after its own device, whatever device the caller is on, has finished its work, and not at all where that is not known."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "place_pool.h"
using namespace bigmac;

static int current = 0, synchronized = -1, answer = 0;
struct Fake {
    static int get(int* device) { *device = current; return 0; }
    static int set(int device) { current = device; return 0; }
    static int synchronize() { synchronized = current; return answer; }
};
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

int main() {
    PlacePool<2, 2> pool;
    CHECK(pool.take(-1) == -1 && pool.take(2) == -1);
    CHECK(pool.take(1) == 0 && pool.take(1) == 1 && pool.take(1) == -1);
    CHECK(pool.take(0) == 0);                                   // a pool of its own on every device
    // a handle of device 1 goes while device 0 is current
    CHECK(pool.give<Fake>(1, 0) && synchronized == 1 && current == 0);
    CHECK(pool.take(1) == 0);
    // device 1 does not say that its work is done
    answer = 1;
    CHECK(!pool.give<Fake>(1, 0) && synchronized == 1 && current == 0);
    CHECK(pool.take(1) == -1);
    answer = 0;
    CHECK(pool.give<Fake>(0, 0) && synchronized == 0 && current == 0);
    pool.give_unused(1, 1);
    CHECK(pool.take(1) == 1);
    { OnDevice<Fake> on(1); CHECK(on.ok && current == 1); }
    CHECK(current == 0);
    return 0;
}
"""


def test_places_go_back_after_their_own_device(tmp_path):
    src = tmp_path / "pool.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "pool"
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "paper_2502_16927_b200", "csrc"), "-o", str(exe), str(src)],
                   check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
