"""The sleep before a poll: a computed sleep of up to 64 ns is spent polling, and the cap shortens a
longer one without turning it into none.  Evaluated by the compiler (no GPU)."""
import os
import subprocess

from paper_1110_4623_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CASES = [(0, 2000, 0), (1, 2000, 0), (64, 2000, 0), (65, 2000, 65), (2000, 2000, 2000), (4000, 2000, 2000),
         (65, 64, 64), (1000, 64, 64), (1000, 32, 32), (1000, 1, 1), (64, 32, 0), (1000, 0, 0),
         (0xFFFFFFFF, 4000, 4000)]


def test_cap_keeps_the_sleep(tmp_path):
    src = tmp_path / "poll_sleep.cu"
    src.write_text('#include <cuda_runtime.h>\n#include "gsync_device.cuh"\n' + "".join(
        f'static_assert(gsync::poll_sleep_ns({ns}u, {cap}u) == {want}u, "{ns} ns, cap {cap}");\n'
        for ns, cap, want in CASES))
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I" + os.path.join(ROOT, "include"), "-c", str(src),
                        "-o", str(tmp_path / "poll_sleep.o")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
