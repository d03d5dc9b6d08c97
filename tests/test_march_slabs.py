"""The block plans of the FP32 plane-marching kernels on tall lattices of few
tiles, on the host: no plan leaves half of the multiprocessors idle while its
slabs could be thinner."""

import os
import subprocess

from paper_2105_00448_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_tall_narrow_lattices_are_cut_thin(tmp_path):
    lib = _build.build()
    exe = str(tmp_path / "march_slabs")
    subprocess.run([_build._nvcc(), *_build.ARCH, "-std=c++17", "-O1", "-I", _build.INCLUDE, "-I", _build.CSRC,
                    os.path.join(HERE, "cuda", "march_slabs.cu"), lib, "-Xlinker", "-rpath=" + os.path.dirname(lib),
                    "-o", exe], check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
