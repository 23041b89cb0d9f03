"""The grid of a launch with one block per item stays within CUDA's limit (2^31 - 1 blocks along x)
for every particle count that bp_smoothing_lengths takes (below 2^32), and is never empty."""
import subprocess

from paper_2201_02632_gb300 import build as B

LIMIT = 2**31 - 1


def test_item_grid_within_the_launch_limit(tmp_path):
    ns = [1, 31, 2**20, LIMIT - 1, LIMIT, 2**31, 2**31 + 1, 2**32 - 1]
    src = tmp_path / "grid.cu"
    src.write_text('#include <cstdio>\n#include "bp_internal.cuh"\nint main() {\n' + "".join(
        f'  std::printf("%u\\n", bp_item_grid({n}LL));\n' for n in ns) + "  return 0;\n}\n")
    exe = tmp_path / "grid"
    r = subprocess.run([B._nvcc(), *B.ARCH, *B.NVFLAGS, "-I", B.CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    assert [int(v) for v in out.stdout.split()] == [min(n, LIMIT) for n in ns]
