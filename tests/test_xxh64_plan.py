"""The launch plan of wm_checksum_xxh64 (csrc/wm_xxh64_plan.h), compiled for the host: every chunk is
some block's, at every number of chunks that the call's 32 bits can hold."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "wm_xxh64_plan.h"
int main(int argc, char** argv)
{
    for (int i = 1; i + 1 < argc; i += 2) {
        const wm::XxhPlan p = wm::xxh64_plan((uint32_t)strtoul(argv[i], nullptr, 10), (uint32_t)strtoul(argv[i + 1], nullptr, 10));
        printf("%d %u %u %u\n", p.paced ? 1 : 0, p.blocks, p.rows, p.rows0);
    }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-Wall", "-I", os.path.join(ROOT, "paper_2607_10389_b200", "csrc"),
                           str(d / "plan.cpp"), "-o", str(d / "plan")])

    def run(n_chunks, n_sm):
        out = subprocess.run([str(d / "plan"), str(n_chunks), str(n_sm)], capture_output=True, text=True)
        assert out.returncode == 0, (n_chunks, n_sm, out.returncode)
        return [int(v) for v in out.stdout.split()]
    return run


@pytest.mark.parametrize("n_sm", [1, 13, 132, 148, 160])
def test_every_chunk_has_a_block(plan, n_sm):
    edges = [1, n_sm, 8 * n_sm, 16 * n_sm, 32 * n_sm, 2 ** 30, 2 ** 32 - 16 * n_sm]
    for n in sorted({e + d for e in edges for d in (-1, 0, 1)} | {2 ** 31, 2 ** 32 - 1}):
        if not 1 <= n < 2 ** 32:
            continue
        paced, blocks, rows, rows0 = plan(n, n_sm)
        assert paced == (n <= 32 * n_sm), n
        if paced:
            assert (blocks - 1) * rows < n <= blocks * rows and blocks <= 2 * n_sm, n      # no block without a chunk
            assert 1 <= rows0 <= 8 and 0 <= rows - rows0 <= min(rows0, 8), n
            assert rows == -(-n // ((1 if n <= 16 * n_sm else 2) * n_sm)), n
        else:
            assert blocks == -(-n // 8) < 2 ** 31, n
