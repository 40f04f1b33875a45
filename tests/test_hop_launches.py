"""How the sampler's hops are cut and launched, by the host code alone: a program that lists the launches needs no GPU."""
import os
import shutil
import subprocess

import pytest

from paper_2202_02365_b200 import build

SOURCE = r"""
#include <cstdio>
#include "mg_sample.cu"

int mg_fail(mg_ctx*, int code, const char*, ...) { return code; }
int mg_cuda_fail(mg_ctx*, cudaError_t, const char*) { return MG_ERR_CUDA; }
void mg_prof_begin(mg_ctx*, int) {}
void mg_prof_end(mg_ctx*, int, int64_t) {}

int main() {   // bound of the hop, a hop, fanout, lists | thread per node, blocks per SM, largest tile, shared memory, tile of the hop
    const int64_t sizes[] = {1, 5000, 18944, 18945, 23680, 37889, 47361, 70000, 75777, 94000, 94721, 128000, 151552, 160000, 500000, 909313, 1000000, 1818624, 2000000, 2000000000};
    for (int64_t bound : sizes)
        for (int f = 1; f <= 33; ++f)
            for (int lists = 1; lists <= 2; ++lists)
                for (int64_t n : sizes) {
                    if (n > bound) break;
                    const HopLaunch l = hop_launch(f, bound, 148, lists == 2, 0);
                    printf("%lld %lld %d %d %d %d %d %zu %d\n", (long long)bound, (long long)n, f, lists, (int)l.thread, l.per_sm, l.tile_cap, l.smem,
                           std::min(hop_tile(n, 148, l.per_sm, l.thread), l.tile_cap));
                }
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    made_in = tmp_path_factory.mktemp("launches")
    source = made_in / "launches.cu"
    source.write_text(SOURCE)
    program = str(made_in / "launches")
    made = subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O0", "-Xptxas", "-O0", "-Xcompiler", "-w",
                           "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"), str(source), "-o", program], capture_output=True, text=True)
    assert made.returncode == 0, made.stderr[-2000:]
    return program


# a hop in tiles of fewer nodes than a block has threads is worked on at once: no more tiles than blocks lie on the SMs together
def test_small_tiles_of_a_hop_are_all_in_work(program):
    ran = subprocess.run([program], capture_output=True, text=True)
    rows = [[int(x) for x in line.split()] for line in ran.stdout.splitlines()]
    assert len(rows) > 10_000 and any(row[4] for row in rows)
    for bound, n, f, lists, thread, per_sm, tile_cap, smem, tile in rows:
        assert 2 <= per_sm <= (4 if thread and f > 2 else 5)      # (what __launch_bounds__ has, 64 registers a thread or 48)
        assert tile >= 256 or -(-n // tile) <= per_sm * 148, (bound, n, f, lists)
        if thread:      # as many blocks as the tiles are cut for lie on an SM, and their shared memory leaves it more than the least L1
            held = min(4 if f > 2 else 5, 228 * 1024 // (smem + 1024 + 144))
            assert held == per_sm and held * (smem + 1024 + 144) <= 196 * 1024, (bound, f, lists)
            assert smem <= 1024 * 36 + 256 * 20 * 2 * 4 + 8 * 4096
        assert -(-n // tile) <= n // 256 + 5 * 148 + 2            # (the tiles' states that a sample has room for)


# a hop that may fill tiles of as many nodes as a block has threads is picked by a thread per node, whatever its fanout of up to twenty and its lists
def test_large_hops_are_picked_by_a_thread_per_node(program):
    ran = subprocess.run([program], capture_output=True, text=True)
    for bound, n, f, lists, thread, *_ in ([int(x) for x in line.split()] for line in ran.stdout.splitlines()):
        assert thread == (bound > 128 * 5 * 148 and f <= 20), (bound, f, lists)
