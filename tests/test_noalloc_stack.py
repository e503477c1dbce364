"""The no-allocation run is meant for plug-ins, whose threads often have small
stacks: its host code keeps no more than a few kilobytes there."""
import os
import subprocess

from paper_2007_07379_gb300 import build


def test_stack_frame(tmp_path):
    src = os.path.join(build.CSRC, "noalloc.cu")
    cmd = [build._nvcc()] + build._flags() + ["-Xcompiler", "-Werror=frame-larger-than=4096", "-c", src,
                                              "-o", str(tmp_path / "noalloc.o")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
