"""Device arithmetic that is plain C++ (host and device functions of the csrc headers), compiled for the host and
compared with wider or plainer arithmetic. No GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2601_02336_gb300", "csrc")


def _run(tmp_path, source, *args, libs=()):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    exe = str(tmp_path / "check")
    cmd = ["g++", "-std=gnu++17", "-O2", "-ffp-contract=off", f"-I{include}", f"-I{CSRC}", "-o", exe,
           os.path.join(ROOT, "tests", source)] + list(libs)
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe] + [str(a) for a in args], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return r.stdout.split(), r.stderr


@pytest.mark.parametrize("seed", [1, 2])
def test_quotient_has_the_bits_of_the_division(tmp_path, seed):
    """quotient(t, c, 1 / c) equals t / c bit for bit: random operands, the edges of the exponent range in which it
    takes the fused steps, zeros of both signs, subnormals, infinities and NaN as numerator and divisor."""
    (n, bad), err = _run(tmp_path, "quotient_check.cpp", seed)
    assert int(n) > 4_000_000 and int(bad) == 0, err
