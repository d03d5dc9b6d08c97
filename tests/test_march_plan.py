"""The block plans of the FP32 plane-marching kernels, on the host: no block
has more segment sums than its shared memory has slots (heights 1 to 300, one
tile to thousands, single lattices and batches), and the blocks cover the
planes.  And on a GPU a lattice of 17 planes with more tiles than blocks
resident at once, in pass A's, the V-cycle's and the residual's kernels."""

import os
import subprocess

import numpy as np
import pytest

from paper_2105_00448_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_segments_fit_their_slots(tmp_path):
    lib = _build.build()
    exe = str(tmp_path / "march_plan")
    subprocess.run([_build._nvcc(), *_build.ARCH, "-std=c++17", "-O1", "-I", _build.INCLUDE, "-I", _build.CSRC,
                    os.path.join(HERE, "cuda", "march_plan.cu"), lib, "-Xlinker", "-rpath=" + os.path.dirname(lib),
                    "-o", exe], check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("precond", ["mg", "jacobi"])
def test_many_tiles_of_17_planes(precond, rng):
    """A step of 1000 x 1000 x 17 sites: the solves' recomputed residuals meet
    their tolerance, and the fields repeat bit for bit."""
    from paper_2105_00448_gb300 import hca
    from synth import make_maps

    nx, ny, nz = 1000, 1000, 17
    maps = make_maps(nx, ny, nz, corr_len=4.0, seed=5)
    pc = hca.HCA_PC_MG if precond == "mg" else hca.HCA_PC_JACOBI
    out = []
    for _ in range(2):
        sim = hca.Sim.create(nx, ny, nz, maps.p_cell, maps.perf, maps.p_vessel, precision="f32", n_drugs=1, seed=5,
                             preconditioner=pc)
        sim.step(1)
        st = sim.stats()
        assert st["o2_rel_residual"] <= 1e-8 and st["drug_rel_residual"][0] <= 1e-8
        out.append((sim.states(), sim.field(hca.FIELD_O2), sim.field(hca.FIELD_DRUG0)))
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
