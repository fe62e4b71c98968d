"""div_markstein (csrc/df64.cuh) equals the FP32 division bit for bit: random
operands over the exponent range it is used in, significands next to 1 and to
2, and quotients near the denormal range. Compiled for the host, where the
reciprocal is the same correctly rounded 1 / b."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_quotients_equal_the_division(tmp_path):
    exe = str(tmp_path / "df64_div_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off",
                           "-I" + os.path.join(ROOT, "paper_1612_07875_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "native", "df64_div_check.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True)
    n, bad = (int(v) for v in out.stdout.split())
    assert out.returncode == 0 and bad == 0 and n > 20_000_000
