"""A push from aligned device memory whose kernel gives up a wait: the row is
reported as timed out, but the snapshot is in its ring slot whole, as after a
separate copy, so that sdmd_rebuild can restore G."""
import os
import subprocess

import pytest

from paper_1612_07875_gb300 import build as B

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("item", [0, 1, 2])
def test_snapshot_is_whole_after_an_expired_wait(item, tmp_path):
    exe = str(tmp_path / "gram_row_expire")
    subprocess.check_call([B.nvcc()] + B.ARCH + ["-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I" + B.INCLUDE, "-I" + B.CSRC,
                           "-DSDMD_GR_WAIT_CYCLES=4000000LL", "-DSDMD_GR_STARVED_ITEM=%d" % item,
                           os.path.join(ROOT, "tests", "native", "gram_row_expire.cu"),
                           os.path.join(B.CSRC, "gram_row.cu"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout
    assert out.stdout.split() == ["1"] * 5
