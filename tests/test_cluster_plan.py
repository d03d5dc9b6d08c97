"""The coarse levels of FP32 hierarchies, on the host: whatever the lattice's
shape, up to the most sites a lattice may have, the levels end at 512 sites or
fewer and some cluster holds the last of them (else a handle would be refused)."""

import os
import subprocess

from paper_2105_00448_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_every_hierarchy_has_a_cluster(tmp_path):
    lib = _build.build()
    exe = str(tmp_path / "cluster_plan")
    subprocess.run([_build._nvcc(), *_build.ARCH, "-std=c++17", "-O1", "-I", _build.INCLUDE, "-I", _build.CSRC,
                    os.path.join(HERE, "cuda", "cluster_plan.cu"), lib, "-Xlinker", "-rpath=" + os.path.dirname(lib),
                    "-o", exe], check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
