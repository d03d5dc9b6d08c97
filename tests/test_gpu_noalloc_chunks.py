"""The allocation-free residual's chunk sizes: one row a chunk below 609 rows,
then growing to 32; row counts on both sides of each change, rows shorter and
longer than a block, against the oracle (same tolerance as the entry point's
other tests)."""

import numpy as np
import pytest

from gpu_helpers import random_states
from oracle import params as Pm
from paper_2105_00448_gb300 import hca
from test_zz_no_alloc import device_arrays, oracle_rel_residual

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 5), (19, 32, 9), (29, 21, 9), (30, 41, 300), (152, 128, 3), (59, 331, 3)])
def test_chunk_sizes(shape, rng):
    nz, ny, nx = shape
    st = random_states(shape, rng)
    st.reshape(-1)[0] = Pm.VESSEL
    K_prev, K = rng.uniform(0.0, 20.0, shape), rng.uniform(0.0, 20.0, shape)
    ref, tol = oracle_rel_residual(st, K_prev, K, Pm.Config(nx=nx, ny=ny, nz=nz))
    args = device_arrays(st, K_prev, K)
    got = [hca.hca_o2_residual_noalloc(hca.make_config(nx, ny, nz), *args) for _ in range(2)]
    assert got[0] == got[1] and abs(got[0] - ref) <= tol
