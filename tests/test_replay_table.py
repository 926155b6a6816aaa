"""Which calls a stage replays from graphs (csrc/replay.h, host code, compiled here with the system's C++ compiler): rounds of more calls than the table
holds still replay as many as it holds, buffers that are no longer used make room, and a call is never mistaken for another."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "replay.h"
using namespace ast;
static std::vector<Replay> table;
static long drops = 0;
// a call as the stage makes it: twice direct, then captured; 1: replayed
static int call(bool bwd, int slot, size_t a, size_t b, uint64_t round) {
    cudaGraphExec_t dropped;
    Replay* r = replay_entry(table, bwd, slot, (const void*)a, (const void*)b, round, &dropped);
    drops += dropped != nullptr;
    if (table.size() > MAX_REPLAYS) exit(2);
    if (!r) return 0;
    if (r->bwd != bwd || r->slot != slot || r->a != (const void*)a || r->b != (const void*)b) exit(3);
    if (!r->exec && r->seen < 2) { ++r->seen; return 0; }
    if (!r->exec) r->exec = (cudaGraphExec_t)(size_t)1;
    return 1;
}
// rounds of M micro-batches, all forwards first, `sets` buffer sets in turn, buffers numbered from `base`; prints how many calls the last `sets` rounds replayed
int main(int argc, char** argv) {
    uint64_t round = 0;
    for (int i = 1; i + 3 < argc; i += 4) {
        const int M = atoi(argv[i]), sets = atoi(argv[i + 1]), base = atoi(argv[i + 2]), rounds = atoi(argv[i + 3]);
        long replayed = 0;
        for (int r = 0; r < rounds; ++r, ++round)
            for (int k = 0; k < 2; ++k)
                for (int m = 0; m < M; ++m) {
                    const size_t buf = 16 * (size_t)(base + (r % sets) * M + m);
                    const int got = call(k == 1, m, buf, buf + 8, round);
                    if (r >= rounds - sets) replayed += got;
                }
        printf("%ld ", replayed);
    }
    printf("%ld\n", drops);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    cuda = "/usr/local/cuda/include"
    if not cxx or not os.path.isdir(cuda):
        pytest.skip("no C++ compiler or CUDA headers")
    d = tmp_path_factory.mktemp("replay")
    src = d / "main.cc"
    src.write_text(MAIN)
    exe = str(d / "main")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2408_08015_b200", "csrc"), "-I", cuda, str(src), "-o", exe], check=True)
    return lambda *a: [int(v) for v in subprocess.run([exe] + [str(v) for v in a], check=True, capture_output=True, text=True).stdout.split()]


@pytest.mark.parametrize("micro, sets", [(1, 1), (8, 1), (32, 1), (33, 1), (40, 1), (200, 1), (8, 4), (8, 5), (1, 40), (3, 64)])
def test_steady_rounds_fill_the_table(program, micro, sets):
    """Every round of a cycle asks for two calls a micro-batch and buffer set."""
    replayed, drops = program(micro, sets, 0, 4 * sets)
    assert replayed == min(2 * micro * sets, 64) and drops == 0


def test_new_buffers_take_the_place_of_old_ones(program):
    a, b, drops = program(32, 1, 0, 4, 32, 1, 1000, 70)
    assert (a, b, drops) == (64, 64, 64)


def test_buffers_used_once_are_never_captured(program):
    replayed, drops = program(4, 500, 0, 500)
    assert replayed == 0 and drops == 0
