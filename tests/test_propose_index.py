"""Index arithmetic of the proposal kernel (csrc/kernels.cuh, propose_task and
propose_blocks) compiled for the host: every electron's coordinates and uniform are
covered once, up to the largest electron count an int holds."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1605_08423_gb300", "csrc")
PROGRAM = r"""
#include <cstdio>
#include "common.cuh"
#include "kernels.cuh"
using namespace qmc;
int main() {
    const int sizes[] = {2, 5, 4096, (1 << 29) - 1, 1 << 29, (1 << 29) + 5, (1 << 30) + 7, 2147483647};
    for (int rows : sizes)
        for (int form = 0; form < 2; ++form) {
            const bool pc = form == 1;
            const int tpb = pc ? 128 : 256;
            const long long threads = (long long)propose_blocks(rows, pc, tpb) * tpb, tasks = (pc ? 4LL : 1LL) * rows;
            if (threads < tasks || threads >= tasks + tpb) return printf("blocks %d %d\n", rows, form), 1;
            auto check = [&](long long k) {      // 3 rows coordinates in order, then rows uniforms
                if (k < 0 || k >= threads) return true;
                const ProposeTask p = propose_task(k, rows, pc);
                if (k >= tasks) return p.t < 0;
                if (pc && k < 3LL * rows) return p.t == k / 3 && p.mu == (int)(k % 3);
                return p.t == (pc ? k - 3LL * rows : k) && p.mu == 3;
            };
            bool ok = true;
            for (long long k = 0; k < threads; k += tasks / 4099 + 1) ok = ok && check(k);
            for (long long d = -8; d < 8; ++d) ok = ok && check(d) && check(3LL * rows + d) && check(tasks + d) && check(2147483648LL + d);
            if (!ok) return printf("task %d %d\n", rows, form), 1;
        }
    puts("ok");
    return 0;
}
"""


def test_every_electron_is_proposed_once(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "index.cu", tmp_path / "index"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-I",
                    os.path.join(CSRC, "..", "..", "include"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
