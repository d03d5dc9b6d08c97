"""Pass A's form for flat lattices against its marching form, bit for bit: a
handle of flat lattices takes the former, a batch in which another lattice has
more planes the latter.  Lattices of one tile and of more than a wave of blocks
holds, ragged rows and one-row lattices; solves of one iteration (nothing
carried over), carried steps, and solves cut off by maxit."""

import numpy as np
import pytest

from oracle import params as Pm
from paper_2105_00448_gb300 import hca
from synth import make_maps

pytestmark = pytest.mark.gpu


def _fields(shapes, pc, **more):
    """States and fields of the first lattice after two steps."""
    cfgs, maps = [], []
    for i, (nz, ny, nx) in enumerate(shapes):
        m = make_maps(nx, ny, nz, corr_len=3.0, seed=20 + i)
        maps.append((m.p_cell, m.perf, m.p_vessel))
        cfgs.append(hca.make_config(nx, ny, nz, precision="f32", n_drugs=1, seed=20 + i, preconditioner=pc, **more))
    sim = hca.Sim(cfgs, maps, batch=True)
    sim.step(2, allow_noconv=True)
    out = [sim.states(0), sim.stats(0)["o2_iterations"], sim.stats(0)["o2_rel_residual"]]
    out += [sim.field(f, 0) for f in (hca.FIELD_O2, hca.FIELD_DRUG0)]
    sim.close()
    return out


@pytest.mark.parametrize("more", [{}, {"maxit": 1, "max_outer": 2}, {"max_outer": 0}], ids=["dc", "maxit1", "plain"])
@pytest.mark.parametrize("pc", [hca.HCA_PC_JACOBI, hca.HCA_PC_MG], ids=["jacobi", "mg"])
@pytest.mark.parametrize("shape", [(1, 40, 60), (1, 27, 129), (1, 1, 700), (1, 700, 1), (1, 700, 1101), (1, 900, 801)])
def test_same_bits_as_the_marching_form(shape, pc, more):
    flat = _fields([shape, (1, 33, 47)], pc, **more)
    march = _fields([shape, (9, 12, 10)], pc, **more)
    for a, b in zip(flat, march):
        assert np.array_equal(a, b)
