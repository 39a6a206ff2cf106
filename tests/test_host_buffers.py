"""The library's decisions about a caller's buffers (csrc/stp_host.h), compiled on
the host: which byte ranges share memory."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_30533_gb300", "csrc")


def _run(tmp_path, body):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include "stp_host.h"\n#include <cstdio>\nint main() {\n%s\nreturn 0;\n}\n' % body)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


# a, bytes, b, bytes: shares a byte?
RANGES = [(64, 16, 80, 16, 0), (80, 16, 64, 16, 0), (64, 17, 80, 16, 1), (64, 16, 64, 16, 1), (64, 100, 70, 1, 1),
          (70, 1, 64, 100, 1), (64, 0, 64, 16, 0), (64, 16, 70, 0, 0), (0, 16, 8, 16, 0), (64, 16, 0, 99, 0)]


@pytest.mark.parametrize("a,na,b,nb,meet", RANGES)
def test_ranges_meet(tmp_path, a, na, b, nb, meet):
    out = _run(tmp_path, 'std::printf("%%d", (int)stp::ranges_meet((void*)%dul, %d, (void*)%dul, %d));' % (a, na, b, nb))
    assert out == [str(meet)]
