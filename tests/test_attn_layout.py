"""The tensor-core attention kernel's shared-memory plans over every k, checked on the host by a program
compiled from the kernel's own header (attn_layout_check.cu)."""
import os
import subprocess

from paper_2106_06899_gb300 import build as B


def test_plans_stay_inside_shared_memory(tmp_path):
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "attn_layout_check.cu")
    exe = str(tmp_path / "attn_layout_check")
    r = subprocess.run([B._nvcc(), "-std=c++17", "-O1", "--expt-relaxed-constexpr", f"-I{B.CSRC}", f"-I{B.INCLUDE}",
                        *B.ARCH, src, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
