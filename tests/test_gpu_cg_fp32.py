"""The FP32 CG passes (marching pass A, streaming pass B, x += alpha p carried
from one iteration to the next) where they can go wrong: lattices of one patch
and of several tiles, row counts around a tile's, padding sites, one-plane
and one-row lattices, solves of one iteration (nothing carried), inner solves
cut off by maxit, and the plain FP32 form without defect correction.

Fields against the FP64 solution of the same system (the oracle's
solver, to 1e-13): FP32 storage of the reaction coefficients
perturbs the system by 2^-24 and the field is rounded once, so with residuals
of 1e-8 the relative error stays below 1e-6 (the bound of the other FP32
tests).
"""

import numpy as np
import pytest

from gpu_helpers import make_pair, random_states
from oracle import multigrid as MG
from oracle import params as Pm
from oracle import stencil as S
from paper_2105_00448_gb300 import hca

pytestmark = pytest.mark.gpu

SHAPES = [(16, 16, 16), (1, 1, 700), (1, 30, 41), (5, 1, 66), (7, 27, 61), (6, 26, 64), (6, 28, 68), (3, 55, 130),
          (40, 9, 7)]


def _solution(st, K_prev, cfg):
    K64 = K_prev.astype(np.float64)
    return MG.mg_pcg(S.o2_coupling(cfg), S.o2_reaction(st, K64, cfg), S.o2_rhs(st, cfg), K64, 1e-13, 1000)[0]


@pytest.mark.parametrize("pc", [hca.HCA_PC_JACOBI, hca.HCA_PC_MG], ids=["jacobi", "mg"])
@pytest.mark.parametrize("shape", SHAPES)
def test_oxygen_solve_matches_fp64(shape, pc, rng):
    sim, cfg, _ = make_pair(shape, "f32", seed=6, n_drugs=0, rtol_o2=1e-8, picard_maxit=1, preconditioner=pc)
    st = random_states(shape, rng)
    st.reshape(-1)[0] = Pm.VESSEL
    K_prev = rng.uniform(0.0, 20.0, shape).astype(np.float32)
    sim.set_states(st)
    sim.set_field(hca.FIELD_O2, K_prev)
    sim.stage(hca.STAGE_O2)
    K, s = sim.field(hca.FIELD_O2), sim.stats()
    sim.close()
    ref = _solution(st, K_prev, cfg)
    assert s["o2_rel_residual"] <= 1e-8
    assert np.max(np.abs(K - ref)) <= 1e-6 * np.max(np.abs(ref))


@pytest.mark.parametrize("pc", [hca.HCA_PC_JACOBI, hca.HCA_PC_MG], ids=["jacobi", "mg"])
def test_inner_solves_cut_off_by_maxit(pc, rng):
    """maxit = 1 and 2: every sweep's correction is one or two iterations (its
    step added by the update alone, or half carried by pass A); the sweeps
    still shrink the residual monotonically."""
    shape = (10, 27, 61)
    st = random_states(shape, rng)
    st.reshape(-1)[0] = Pm.VESSEL
    K_prev = rng.uniform(0.0, 20.0, shape).astype(np.float32)
    rel = {}
    for maxit in (1, 2):
        for outer in (1, 4):
            sim, _, _ = make_pair(shape, "f32", seed=6, n_drugs=0, rtol_o2=1e-12, picard_maxit=1, preconditioner=pc,
                                  maxit=maxit, max_outer=outer)
            sim.set_states(st)
            sim.set_field(hca.FIELD_O2, K_prev)
            sim.stage(hca.STAGE_O2, allow_noconv=True)
            s = sim.stats()
            assert s["o2_iterations"] == maxit * outer
            rel[maxit, outer] = s["o2_rel_residual"]
            sim.close()
    assert rel[2, 1] < rel[1, 1] and rel[1, 4] < rel[1, 1] and rel[2, 4] < rel[2, 1]


@pytest.mark.parametrize("pc", [hca.HCA_PC_JACOBI, hca.HCA_PC_MG], ids=["jacobi", "mg"])
def test_plain_fp32_solve(pc, rng):
    """max_outer = 0: no defect correction, x updated by pass B; converges to
    the FP32 residual floor's neighbourhood (rtol 1e-4)."""
    shape = (9, 27, 61)
    sim, cfg, _ = make_pair(shape, "f32", seed=6, n_drugs=0, rtol_o2=1e-4, picard_maxit=1, preconditioner=pc,
                            max_outer=0)
    st = random_states(shape, rng)
    st.reshape(-1)[0] = Pm.VESSEL
    K_prev = rng.uniform(0.0, 20.0, shape).astype(np.float32)
    sim.set_states(st)
    sim.set_field(hca.FIELD_O2, K_prev)
    sim.stage(hca.STAGE_O2)
    K = sim.field(hca.FIELD_O2).astype(np.float64)
    sim.close()
    c, a, b = S.o2_coupling(cfg), S.o2_reaction(st, K_prev.astype(np.float64), cfg), S.o2_rhs(st, cfg)
    res = b - S.apply_operator(K, c, a)
    assert np.linalg.norm(res) <= 2e-4 * np.linalg.norm(b)
