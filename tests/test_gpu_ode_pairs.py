"""The per-cell ODEs at the cell counts where the FP32 batches (two cells a
lane) change form: none, one, around half a batch and a batch per warp, with
sites of zero oxygen (no p53 decay) among them, sparse and dense.  Bound: that
of the full-lattice ODE test (FP32 RK4 against the FP64 oracle)."""

import numpy as np
import pytest

from gpu_helpers import make_pair
from oracle import params as Pm
from oracle.odes import ode_update
from paper_2105_00448_gb300 import hca

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("cells", [0, 1, 31, 32, 33, 63, 64, 65, 127, 128, 260])
def test_cell_counts(cells, precision, rng):
    shape = (1, 2, 130)
    sim, cfg, _ = make_pair(shape, precision, seed=7, n_drugs=1, picard_maxit=1)
    st = np.zeros(shape, np.uint8)
    at = rng.permutation(st.size)[:cells]
    st.reshape(-1)[at] = rng.choice([Pm.PROLIF, Pm.QUIESC, Pm.STROMA], cells)
    K = rng.uniform(0.0, 20.0, shape)
    K.reshape(-1)[at[::5]] = 0.0
    fields = {hca.FIELD_O2: K, hca.FIELD_PHI: rng.random(shape), hca.FIELD_P53: 0.1 * rng.random(shape),
              hca.FIELD_VEGFC: 0.3 * rng.random(shape)}
    sim.set_states(st)
    for bit, v in fields.items():
        sim.set_field(bit, v)
    f = {b: sim.field(b).astype(np.float64) for b in fields}
    sim.stage(hca.STAGE_ODE)
    ref = ode_update(st, f[hca.FIELD_PHI], f[hca.FIELD_P53], f[hca.FIELD_VEGFC], f[hca.FIELD_O2], cfg)
    for bit, r in zip((hca.FIELD_PHI, hca.FIELD_P53, hca.FIELD_VEGFC), ref):
        got = sim.field(bit).astype(np.float64)
        rel = np.max(np.abs(got - r) / np.maximum(np.abs(r), 1e-3 * np.max(np.abs(r))))
        assert rel <= (1e-12 if precision == "f64" else 2e-6), (bit, rel)
    sim.close()
