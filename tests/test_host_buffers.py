"""The library's decisions about a caller's buffers (csrc/stp_host.h), compiled on
the host: which byte ranges share memory, and which memory only a copy reaches."""
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


# On a GPU, its number, the current one: another GPU's? Host memory reports an owner too.
@pytest.mark.parametrize("gpu,owner,current,other", [(1, 0, 0, 0), (1, 1, 0, 1), (1, 0, 1, 1), (0, 0, 1, 0), (0, -2, 0, 0)])
def test_other_gpu(tmp_path, gpu, owner, current, other):
    out = _run(tmp_path, 'std::printf("%%d", (int)stp::on_other_gpu(%d, %d, %d));' % (gpu, owner, current))
    assert out == [str(other)]


def test_kernels_take_no_other_gpus_buffers():
    """Every place that hands a caller's pointer to a kernel where a copy used to go asks first."""
    api, mlp = (open(os.path.join(CSRC, f)).read() for f in ("stp_api.cu", "stp_mlp.cu"))
    for src, pointers in ((api, ("min_clearance", "n_checks")), (mlp, ("src", "Y"))):
        for p in pointers:
            assert "other_gpu(%s)" % p in src
