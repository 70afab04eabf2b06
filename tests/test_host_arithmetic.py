"""Device arithmetic that is plain C++ (host and device functions of the csrc headers), compiled for the host and
compared with wider or plainer arithmetic. No GPU."""
import os
import platform
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


@pytest.mark.parametrize("seed", [1, 2])
def test_fixed_point_functions(tmp_path, seed):
    """fixed.cuh's fraction of a turn, sine and cosine of the rest, carrier and moment sums against 113-bit arithmetic,
    each within the bound that the check derives, index wraps, the rest's ends and limb boundaries included."""
    out, _ = _run(tmp_path, "fixed_point_check.cpp", seed, libs=["-lquadmath"] if platform.machine() == "x86_64" else [])
    rows = {out[i]: (float(out[i + 1]), float(out[i + 2])) for i in range(0, len(out), 3)}
    assert set(rows) == {"limbs", "frac", "index_and_rest", "sine", "cosine", "carrier", "carrier_rms_per_part",
                         "moment_per_product", "moment_of_one_per_product"}
    for name, (worst, bound) in rows.items():
        assert worst <= bound, name
