"""The colour sweeps in one launch (a warp per committed cell, cells of every
replicate together) where that form can go wrong: every cell committing at
once (several cells a warp), none (all colours empty), equal K everywhere
(the first free neighbour wins), infinite and NaN K (chosen only by coming
first in scan order), and batches of more replicates than lanes.  The
per-colour launches (HCA_CA_COOP=0), one thread a cell, decide the same.
"""

import numpy as np
import pytest

from gpu_helpers import make_pair, random_states
from paper_2105_00448_gb300 import hca
from synth import make_maps

pytestmark = pytest.mark.gpu


def _both(run, monkeypatch):
    out = []
    for coop in ("1", "0"):
        monkeypatch.setenv("HCA_CA_COOP", coop)
        out.append(run())
    return out


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("commit", [0.0, 0.02, 1.0], ids=["none", "few", "all"])
@pytest.mark.parametrize("field", ["random", "ties", "special"])
@pytest.mark.parametrize("shape", [(1, 1, 7), (1, 40, 33), (30, 31, 90)])
def test_one_launch_equals_per_colour_launches(shape, field, commit, precision, monkeypatch):
    rng = np.random.default_rng(3)
    st = random_states(shape, rng)
    phi = np.where(rng.random(shape) < commit, 1.0 + 0.1 * rng.random(shape), 0.5)
    K = {"random": rng.uniform(0, 20, shape), "ties": np.full(shape, 5.0),
         "special": rng.choice([0.0, -0.0, 3.0, np.inf, -np.inf, np.nan], shape)}[field]
    G = rng.uniform(0, 0.6, shape)

    def run():
        sim, _, _ = make_pair(shape, precision, seed=12, n_drugs=1, picard_maxit=1)
        sim.set_states(st)
        sim.set_field(hca.FIELD_O2, K)
        sim.set_field(hca.FIELD_PHI, phi)
        sim.set_field(hca.FIELD_DRUG0, G)
        sim.stage(hca.STAGE_CA)
        s = sim.stats()
        out = sim.states(), sim.field(hca.FIELD_PHI), [s[k] for k in ("committed", "kills", "divisions", "blocked")]
        sim.close()
        return out

    a, b = _both(run, monkeypatch)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2] == b[2]
    assert a[2][0] == sum(a[2][1:])


def test_many_replicates_in_one_launch(monkeypatch):
    def run():
        cfgs, maps = [], []
        for r in range(40):
            nz, ny, nx = 4 + r % 5, 5 + r % 7, 6 + r % 11
            m = make_maps(nx, ny, nz, corr_len=2.0, seed=r)
            maps.append((m.p_cell, m.perf, m.p_vessel))
            cfgs.append(hca.make_config(nx, ny, nz, precision="f32", n_drugs=1, seed=r, T_cycle=300.0))
        sim = hca.Sim(cfgs, maps, batch=True)
        sim.step(2)
        out = [(sim.states(r), sim.stats(r)["kills"], sim.stats(r)["divisions"]) for r in range(40)]
        sim.close()
        return out

    a, b = _both(run, monkeypatch)
    assert sum(x[2] for x in a) > 0
    for x, y in zip(a, b):
        assert np.array_equal(x[0], y[0]) and x[1:] == y[1:]
