"""Chunk lengths of a batch's matrices (chunks.hpp, host code): the task results of
one matrix, 24 bytes a task of 32 chunks, stay small whatever n."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2501_15126_gb300", "csrc")
MAIN = """
#include "chunks.hpp"
#include <cstdio>
int main() {
    for (int n = 9; n <= 48; ++n) std::printf("%d ", perm::batch_default_chunk_log2(n));
    for (int h = 0; h <= 47; ++h) std::printf("%d ", perm::shared_chunk_log2(h, perm::kBatchTasksLog2));
}
"""


@pytest.fixture(scope="module")
def chunks(tmp_path_factory):
    d = tmp_path_factory.mktemp("chunks")
    (d / "main.cpp").write_text(MAIN)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")])
    v = [int(x) for x in subprocess.check_output([str(d / "main")], text=True).split()]
    return dict(zip(range(9, 49), v[:40])), dict(zip(range(48), v[40:]))


def test_chained_walks(chunks):
    for n, K in chunks[0].items():   # 2^(n-1-K-5) tasks: at most 2^12, or what 2^12 steps a chunk give
        assert 9 <= K <= 12
        assert n - 6 - K <= max(12, n - 18)


def test_eliminated_walks(chunks):
    for h, K in chunks[1].items():   # 2^(h-K-5) tasks: at most 1.5 MB
        assert 0 <= K <= h
        assert h - K - 5 <= 16
        if 5 <= h <= 24:             # measured sizes: 2^3 outer steps a lane where full warps remain
            assert K == min(3, h - 5)
