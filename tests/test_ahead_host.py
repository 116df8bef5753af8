"""Host-side rules of the draw-ahead form (csrc/ahead.h) and of the memory it works in,
compiled with the host compiler and run without a GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1007_3726_gb300", "csrc")


def _cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(d, "cuda_runtime.h")):
        pytest.skip("CUDA headers not found")
    return d


def _run(tmp_path, source, *files):
    """Compiles a C++ program against the library's headers (and some of its files) and
    returns what it prints."""
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(source)
    cmd = ["g++", "-std=c++17", "-g", "-fsanitize=undefined", "-fno-sanitize-recover=undefined", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I",
           _cuda_include(), "-o", str(exe), str(src)]
    for f in files:
        cmd += ["-x", "c++", os.path.join(CSRC, f)]
    r = subprocess.run([*cmd, "-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    return r.stdout


DRAW_GRID = r"""
#include "ahead.h"
#include <cstdio>
using namespace ising;
int main()
{
    const uint32_t T = 512;
    for (uint32_t sms = 1; sms <= 152; sms += sms < 70 ? 1 : 41)
        for (uint32_t L : {320u, 512u})
            for (uint32_t slots : {0u, 1u, 7u, 64u, 128u})
                for (uint32_t tickets : {0u, 1u, 200u, 8192u}) {
                    const uint32_t runs = L * (L / 64) / 2, per = (runs + 31u) & ~31u;
                    const DrawGrid g = draw_grid(sms, T, slots, runs, tickets);
                    // the kernel's loop: CTA c < count_ctas takes items c T + thread, in strides of count_ctas T
                    uint64_t done = 0;
                    for (uint32_t c = 0; c < g.grid && c < g.count_ctas; ++c)
                        for (uint64_t first = (uint64_t)c * T; first < (uint64_t)slots * per; first += (uint64_t)g.count_ctas * T)
                            done += std::min<uint64_t>(T, (uint64_t)slots * per - first);
                    if (done != (uint64_t)slots * per || g.grid < 1 || g.grid > sms) {
                        std::printf("sms %u L %u slots %u tickets %u: %llu of %llu counted by %u of %u CTAs\n", sms, L, slots, tickets,
                                    (unsigned long long)done, (unsigned long long)slots * per, g.grid, g.count_ctas);
                        return 1;
                    }
                }
    return 0;
}
"""


def test_every_snapshot_is_counted_on_any_number_of_sms(tmp_path):
    _run(tmp_path, DRAW_GRID)
