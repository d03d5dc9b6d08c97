"""The defect-correction residual sweep where it can go wrong: lattices of one
patch and of several tiles, padding sites, one-plane and one-row lattices, and
fields whose squares leave the FP32 range (the sums run at a moving scale).

One correction of one iteration, then the reported relative residual against
the residual of the downloaded field in FP64.  The download drops the low word
(2^-24 of a site) and the reaction coefficient and right-hand side are rounded
to FP32, so the norms differ by at most 2^-22 |d K| / |b|; the sums themselves
are good to 1e-6.
"""

import numpy as np
import pytest

from gpu_helpers import make_pair, random_states
from oracle import params as Pm
from oracle import stencil as S
from paper_2105_00448_gb300 import hca

pytestmark = pytest.mark.gpu

SHAPES = [(16, 16, 16), (1, 1, 700), (1, 30, 41), (5, 1, 66), (7, 27, 61), (6, 28, 68), (3, 55, 130), (40, 9, 7)]


@pytest.mark.parametrize("size", [1.0, 1e-21, 1e15])
@pytest.mark.parametrize("pc", [hca.HCA_PC_JACOBI, hca.HCA_PC_MG], ids=["jacobi", "mg"])
@pytest.mark.parametrize("shape", SHAPES)
def test_reported_residual(shape, pc, size, rng):
    K0 = 20.0 * size
    sim, cfg, _ = make_pair(shape, "f32", seed=6, n_drugs=0, rtol_o2=1e-12, picard_maxit=1, preconditioner=pc,
                            maxit=1, max_outer=1, K0=K0)
    st = random_states(shape, rng)
    st.reshape(-1)[0] = Pm.VESSEL
    K_prev = (size * rng.uniform(0.0, 20.0, shape)).astype(np.float32)
    sim.set_states(st)
    sim.set_field(hca.FIELD_O2, K_prev)
    sim.stage(hca.STAGE_O2, allow_noconv=True)
    K, s = sim.field(hca.FIELD_O2).astype(np.float64), sim.stats()
    sim.close()
    c, a, b = S.o2_coupling(cfg), S.o2_reaction(st, K_prev.astype(np.float64), cfg), S.o2_rhs(st, cfg)
    nb = np.linalg.norm(b)
    rel = np.linalg.norm(b - S.apply_operator(K, c, a)) / nb
    tol = 1e-6 * rel + 2.0**-22 * np.linalg.norm((6.0 * c + a) * K) / nb
    assert abs(s["o2_rel_residual"] - rel) <= tol
