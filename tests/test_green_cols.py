"""The FP64 z pass's columns per block (csrc/green_cols.h), compiled for the host, against
the times of whole sweeps with each width."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_00822_gb300", "csrc")

# (nx, ny, nz, members): us a sweep on a GB300 (152 SMs) with 4, 2 and 1 columns
MEASURED = {
    (16, 16, 16, 1): (30.1, 30.2, 30.4), (24, 24, 24, 1): (37.2, 38.2, 37.0), (32, 32, 32, 1): (51.5, 43.3, 44.0),
    (48, 48, 48, 1): (128.1, 122.5, 125.5), (64, 64, 64, 1): (241.3, 240.2, 249.3),
    (96, 96, 96, 1): (989.9, 947.5, 1003.7), (128, 128, 128, 1): (1940.8, 1880.7, 1941.8),
    (192, 192, 192, 1): (7065.6, 6981.7, 7175.0), (256, 256, 256, 1): (16406.3, 16059.5, 16168.5),
    (32, 32, 32, 4): (138.6, 121.8, 126.2), (48, 96, 24, 1): (137.4, 133.6, 131.6),
    (24, 64, 32, 1): (67.3, 64.4, 66.3), (64, 64, 32, 1): (124.2, 129.1, 127.0),
    (32, 48, 96, 1): (178.6, 158.8, 170.3), (24, 32, 128, 1): (117.2, 117.8, 111.5),
    (32, 32, 32, 16): (423.5, 414.3, 414.0), (64, 64, 64, 8): (1677.3, 1621.8, 1743.5),
    (24, 24, 24, 8): (127.8, 122.9, 126.7), (96, 48, 96, 2): (947.9, 908.9, 962.1),
    (24, 48, 16, 1): (38.1, 37.5, 38.3), (48, 24, 16, 1): (45.1, 44.6, 43.8), (16, 32, 48, 1): (47.5, 47.6, 41.4),
    (48, 48, 24, 1): (81.1, 73.7, 69.4), (96, 64, 48, 1): (310.2, 306.0, 342.2),
    (32, 64, 64, 1): (153.5, 128.3, 140.8), (128, 32, 32, 1): (124.8, 130.4, 127.3),
    (64, 48, 32, 1): (117.8, 114.6, 114.1), (24, 24, 24, 3): (57.1, 60.9, 61.7), (32, 24, 48, 2): (86.8, 79.4, 89.2),
    (16, 16, 16, 20): (88.7, 85.8, 88.6), (48, 32, 24, 2): (95.6, 95.6, 95.1),
    (192, 48, 24, 1): (211.2, 232.9, 232.8), (64, 32, 32, 2): (118.4, 123.2, 121.3),
    (16, 24, 64, 1): (52.3, 44.4, 42.5), (96, 24, 24, 1): (85.0, 70.6, 73.4), (128, 64, 64, 1): (461.7, 440.1, 476.4),
    (96, 96, 48, 1): (461.8, 452.0, 505.3),
}


def test_chosen_widths_are_close_to_the_fastest(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "cols.cpp"
    src.write_text('#include "green_cols.h"\n#include <cstdio>\nint main() { int nx, ny, b; while (std::scanf("%d %d %d", '
                   '&nx, &ny, &b) == 3) std::printf("%d\\n", bfcs::green_cols_fp64(nx / 2 + 1, ny, b, 152)); }\n')
    exe = tmp_path / "cols"
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True, timeout=120)
    asked = "".join(f"{nx} {ny} {b}\n" for nx, ny, _, b in MEASURED)
    got = subprocess.run([str(exe)], input=asked, capture_output=True, text=True, check=True, timeout=60).stdout.split()
    loss = [dict(zip((4, 2, 1), times))[int(cols)] / min(times) for times, cols in zip(MEASURED.values(), got, strict=True)]
    assert max(loss) <= 1.05, dict(zip(MEASURED, loss))
    assert np.exp(np.log(loss).mean()) <= 1.01
