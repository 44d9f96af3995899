"""The share of the device that optional vectors may hold (opt_share in csrc/internal.cuh), on the
host: a quarter of the device for all, a quarter of what is free for one request."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda/include"
GB = 1 << 30

# want, own, held, free, total (GB): allowed?
CASES = [(10, 0, 0, 250, 280, True), (70, 0, 0, 280, 280, True), (71, 0, 0, 280, 280, False),
         (120, 0, 0, 270, 280, False), (10, 0, 61, 200, 280, False), (10, 5, 65, 200, 280, True),
         (10, 0, 20, 39, 280, False), (10, 0, 20, 40, 280, True), (10, 4, 20, 36, 280, True), (1, 0, 0, 0, 280, False)]


@pytest.mark.skipif(not (os.path.isdir(CUDA) and shutil.which("g++")), reason="no CUDA headers or compiler")
def test_share(tmp_path):
    src = '#include "internal.cuh"\n#include <cstdio>\n#include <cstdlib>\nint main(int c, char **v) { size_t a[5];\n' \
          'for (int i = 0; i < 5; ++i) a[i] = strtoull(v[1 + i], 0, 10);\n' \
          'return cgk::opt_share(a[0], a[1], a[2], a[3], a[4]) ? 1 : 0; }\n'
    (tmp_path / "t.cc").write_text(src)
    subprocess.run(["g++", "-std=c++17", "-I" + CUDA, "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_1409_0001_gb300", "csrc"), str(tmp_path / "t.cc"), "-o",
                    str(tmp_path / "t")], check=True)
    for *args, ok in CASES:
        r = subprocess.run([str(tmp_path / "t")] + [str(a * GB) for a in args])
        assert (r.returncode == 1) == ok, args
