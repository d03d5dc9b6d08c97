"""FP64 Jacobi-PCG solves in one launch (small lattices) at the edges of that
form: a few sites, one block, several blocks of one and of two 2-site groups
a thread, lattices just inside and outside its limit (about 300 000 sites),
rows with padding, maxit cut-offs, and batches that mix both forms or need
several rounds of blocks.

The recomputed residual of a solve that stopped at rtol may exceed it only by
the recurrences' drift (a few hundred roundings of 1e-16): 1e-3 rtol is
allowed at rtol = 1e-10.  A batch gives every replicate its own bits.
"""

import numpy as np
import pytest

from gpu_helpers import make_pair, random_states
from oracle import params as Pm
from oracle import stencil as S
from paper_2105_00448_gb300 import hca
from synth import make_maps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 3), (2, 3, 5), (7, 9, 17), (16, 16, 16), (48, 48, 48), (53, 54, 55),
                                   (66, 67, 68), (70, 70, 70), (1, 300, 999)])
def test_solves_reach_their_residual(shape, rng):
    rtol = 1e-10
    sim, cfg, _ = make_pair(shape, "f64", seed=4, n_drugs=1, rtol_o2=rtol, rtol_drug=rtol, picard_maxit=1)
    st = random_states(shape, rng)
    st.reshape(-1)[0] = Pm.VESSEL
    K_prev, G = rng.uniform(0.0, 20.0, shape), rng.random(shape)
    sim.set_states(st)
    sim.set_field(hca.FIELD_O2, K_prev)
    sim.set_field(hca.FIELD_DRUG0, G)
    sim.stage(hca.STAGE_O2)
    K, s = sim.field(hca.FIELD_O2), sim.stats()
    sim.close()
    c, a, b = S.o2_coupling(cfg), S.o2_reaction(st, K_prev, cfg), S.o2_rhs(st, cfg)
    rel = np.linalg.norm(b - S.apply_operator(K, c, a)) / np.linalg.norm(b)
    assert rel <= 1.001 * rtol and abs(rel - s["o2_rel_residual"]) <= 1e-3 * rtol
    assert s["o2_iterations"] > 0


@pytest.mark.parametrize("maxit", [1, 2, 5])
def test_maxit_stops_a_solve(maxit, rng):
    shape = (12, 13, 14)
    sim, _, _ = make_pair(shape, "f64", seed=4, n_drugs=0, rtol_o2=1e-12, picard_maxit=1, maxit=maxit)
    sim.set_field(hca.FIELD_O2, rng.uniform(0.0, 20.0, shape))
    assert sim.stage(hca.STAGE_O2, allow_noconv=True) == hca.HCA_ERR_NOCONV
    assert sim.stats()["o2_iterations"] == maxit
    sim.close()


@pytest.mark.parametrize("sizes", [[(8, 9, 10), (72, 72, 72), (20, 21, 22)], [(40, 40, 40)] * 4 + [(5, 6, 7)] * 8],
                         ids=["mixed", "rounds"])
def test_batches_give_every_replicate_its_own_bits(sizes):
    params = dict(n_drugs=1, rtol_o2=1e-8, rtol_drug=1e-8, picard_tol=1e-6)
    cfgs, maps = [], []
    for r, (nz, ny, nx) in enumerate(sizes):
        m = make_maps(nx, ny, nz, corr_len=3.0, seed=40 + r)
        maps.append((m.p_cell, m.perf, m.p_vessel))
        cfgs.append(hca.make_config(nx, ny, nz, precision="f64", seed=40 + r, **params))
    batch = hca.Sim(cfgs, maps, batch=True)
    batch.step(2)
    for r in range(len(sizes)):
        one = hca.Sim(cfgs[r], maps[r])
        one.step(2)
        assert np.array_equal(batch.states(r), one.states())
        assert np.array_equal(batch.field(hca.FIELD_O2, r), one.field(hca.FIELD_O2))
        assert np.array_equal(batch.field(hca.FIELD_DRUG0, r), one.field(hca.FIELD_DRUG0))
        assert batch.stats(r)["drug_iterations"] == one.stats()["drug_iterations"]
        one.close()
    batch.close()
