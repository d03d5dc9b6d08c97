"""The plane-marching kernels on lattices of more tiles than blocks are resident
at once, so that a block's slab holds several reduction segments (the last one
partial): the V-cycle and the defect correction's residual sweep against the
oracle.  Checks and bounds are those of the smaller shapes."""

import pytest

import test_gpu_dc_residual as R
import test_gpu_march as M
from paper_2105_00448_gb300 import hca

pytestmark = pytest.mark.gpu

SHAPES = [(17, 480, 640), (39, 300, 401), (131, 160, 200)]


@pytest.mark.parametrize("shape", SHAPES)
def test_vcycle(shape, rng, monkeypatch):
    M.test_fp32_vcycle_matches_oracle_and_itself(shape, rng, monkeypatch)


@pytest.mark.parametrize("pc", [hca.HCA_PC_JACOBI, hca.HCA_PC_MG], ids=["jacobi", "mg"])
@pytest.mark.parametrize("shape", SHAPES)
def test_residual(shape, pc, rng):
    R.test_reported_residual(shape, pc, 1.0, rng)
