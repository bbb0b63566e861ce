"""Shared memory of a packed replay launch, computed on the host (no GPU): the same for any order of
its jobs, and never more than the kernel's bound."""
import os
import shutil
import subprocess

import pytest

from paper_2211_17263_gb300 import build, capi

SOURCE = r"""
#include <cstdio>
#include <cstring>
#include "internal.h"
using namespace prdpt;
static TraceJob job(int R, int stride, int pixels, int depth, bool moves, bool black) {
    TraceJob J;
    std::memset(&J, 0, sizeof J);
    J.R = R; J.gstride = stride; J.depth = depth; J.n_var = moves; J.black = black; J.var_mats = 1u;
    J.bw = pixels; J.bh = 1; J.parts = 1; J.chunks = 1; J.emit = 1;
    return J;
}
int main() {
    const int R[] = {2, 8, 10, 24, 32}, px[] = {1, 2, 4, 8, 32}, depth[] = {1, 8, 64};
    for (int moves = 0; moves < 2; ++moves)
        for (int a = 0; a < 75; ++a)
            for (int b = 0; b < 75; ++b) {
                const TraceJob A = job(R[a % 5], 3, px[a / 5 % 5], depth[a / 25], moves, true);
                const TraceJob B = job(R[b % 5], 3, px[b / 5 % 5], depth[b / 25], moves, true);
                TraceLaunch L, M;
                std::memset(&L, 0, sizeof L);
                std::memset(&M, 0, sizeof M);
                replay_cover(L, A); replay_cover(L, B);
                replay_cover(M, B); replay_cover(M, A);
                if (replay_smem(L) != replay_smem(M) || L.pool != M.pool || replay_smem(L) > 160 * 1024 ||
                    L.pool < replay_path_granules(64 * (a / 25 == 2 || b / 25 == 2), moves != 0)) {
                    std::printf("jobs %d %d: %zu and %zu bytes\n", a, b, replay_smem(L), replay_smem(M));
                    return 1;
                }
            }
    return 0;
}
"""


def test_pool_does_not_depend_on_the_order_of_jobs(tmp_path):
    lib = capi.load()._name
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    src, exe = tmp_path / "cover.cpp", tmp_path / "cover"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", f"-I{build.CSRC}", f"-I{cuda}", str(src), lib, "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True,
                         env=dict(os.environ, LD_LIBRARY_PATH=os.path.dirname(lib)))
    assert res.returncode == 0, res.stdout + res.stderr
