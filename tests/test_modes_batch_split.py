"""How a batch of eigensolvers is split into one-CTA and cluster launches: the
CTAs a job runs on also size its shared memory, whatever the job says about
running alone, and embedded complex windows and bad counts are refused. Runs
on the host against the built objects."""
import os
import subprocess

from paper_1612_07875_gb300 import build as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_split_and_sizes_agree(tmp_path):
    objs = [os.path.join(B.BUILD, os.path.basename(s)[:-3] + ".o") for s in B.sources()]
    B.build(force=not all(os.path.exists(o) for o in objs))
    exe = str(tmp_path / "modes_split_check")
    subprocess.check_call([B.nvcc()] + B.ARCH + ["-std=c++17", "--expt-relaxed-constexpr", "-I" + B.INCLUDE, "-I" + B.CSRC,
                           os.path.join(ROOT, "tests", "native", "modes_split_check.cu")] + objs + ["-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout + out.stderr
    tried, bad = (int(v) for v in out.stdout.split())
    assert tried > 2000 and bad == 0
