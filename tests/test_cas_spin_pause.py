"""The CAS spin lock's pause between two attempts: none below 680 blocks and none for the first four
attempts, then the pace of a full atomic unit; what a grid of more blocks than can be resident, or
one spread over many locks, calls for is reached only by a waiter that goes on failing.  Evaluated by
the compiler (no GPU)."""
import os
import subprocess

from paper_1110_4623_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# (blocks, failed attempts, pause)
CASES = [(1, 5, 0), (679, 1000, 0), (680, 4, 0), (680, 5, 42), (680, 10000, 42), (700, 5, 55), (1184, 0, 0), (1184, 4, 0),
         (1184, 5, 367), (1184, 0xFFFFFFFF, 367), (1216, 5, 380), (2400, 5, 380), (2400, 100, 800), (2400, 145, 1160),
         (2400, 1000, 1160), (4864, 5, 380), (4864, 48, 384), (4864, 1000, 2759), (20000, 4, 0), (20000, 5, 380),
         (20000, 499, 3992), (20000, 500, 4000), (20000, 0xFFFFFFFF, 4000), (0xFFFFFFFF, 5, 380),
         (0xFFFFFFFF, 0x20000001, 4000)]


def test_pause(tmp_path):
    src = tmp_path / "pause.cu"
    src.write_text('#include <cuda_runtime.h>\n#include "gsync_device.cuh"\n' + "".join(
        f'static_assert(gsync::cas_spin_pause_ns(gsync::cas_spin_most_ns({b}u), {n}u) == {want}u, "{b} blocks, {n}");\n'
        for b, n, want in CASES))
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I" + os.path.join(ROOT, "include"), "-c", str(src),
                        "-o", str(tmp_path / "pause.o")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
