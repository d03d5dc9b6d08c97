"""Handles whose solves never launch the CG passes do not time them at
creation: the launch shape follows the lattices (the same for every handle),
and HCA_NO_TUNE changes neither it nor the number of kernels launched.  A
lattice too large for the one-launch solve, and multigrid, still time them."""

import pytest

from gpu_helpers import make_pair
from paper_2105_00448_gb300 import hca

pytestmark = pytest.mark.gpu


def _created(shape, no_tune, monkeypatch, **params):
    monkeypatch.setenv("HCA_NO_TUNE", no_tune)
    sim, _, _ = make_pair(shape, "f64", seed=4, n_drugs=1, **params)
    out = (hca.hca_get_launch_config(sim.handle)[0], sim.launches())
    sim.close()
    return out


@pytest.mark.parametrize("shape", [(16, 16, 16), (48, 48, 48), (64, 64, 64)])
def test_one_launch_solves_are_not_timed(shape, monkeypatch):
    tuned, fixed = _created(shape, "0", monkeypatch), _created(shape, "1", monkeypatch)
    assert tuned == fixed and tuned[0] == 512


@pytest.mark.parametrize("shape,params", [((72, 72, 72), {}), ((24, 24, 24), {"preconditioner": hca.HCA_PC_MG})])
def test_solves_by_passes_are_timed(shape, params, monkeypatch):
    tuned, fixed = _created(shape, "0", monkeypatch, **params), _created(shape, "1", monkeypatch, **params)
    assert tuned[1] > fixed[1] and fixed[0] == 128
