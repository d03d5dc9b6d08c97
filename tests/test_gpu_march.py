"""The FP32 multigrid V-cycle's fused forms -- the plane-marching sweeps of
the lattice and the grid levels, and the coarse levels in a thread-block
cluster -- against the FP64 oracle, and bit for bit against themselves with
the levels split between the two in other ways (HCA_MG_CLUSTER: blocks per
cluster, which also moves the first level the cluster holds).

Tolerance of z = M r: storing the diagonal d = c n + a in FP32 perturbs the
reaction a by up to 2^-24 d, and the coarse levels see a smooth error through
the mean reaction, so the relative error is of the order of 2^-24 max(d) /
mean(a); 8 such units are allowed (for the rest of the FP32 arithmetic).
"""

import numpy as np
import pytest

from gpu_helpers import make_pair, random_states
from oracle import multigrid as MG
from oracle import stencil as S
from paper_2105_00448_gb300 import hca

pytestmark = pytest.mark.gpu

# (nz, ny, nx): tiles of one group and of several (16 groups by 12 row pairs
# at most), one more or less than a tile, odd extents on every axis, flat and
# thin lattices, planes along y in the cluster, a chain
SHAPES = [(16, 16, 16), (17, 23, 31), (33, 49, 65), (64, 64, 64), (13, 24, 130), (8, 20, 300), (3, 40, 260),
          (1, 100, 500), (2, 2, 400), (300, 3, 3), (9, 50, 263), (1, 1, 5000)]


def _system(which, st, K, perf, cfg):
    if which == 0:
        return S.o2_coupling(cfg), S.o2_reaction(st, K, cfg)
    return S.drug_coupling(cfg, 0), S.drug_reaction(st, perf, cfg, 0)


@pytest.mark.parametrize("shape", SHAPES)
def test_fp32_vcycle_matches_oracle_and_itself(shape, rng, monkeypatch):
    st = random_states(shape, rng)
    K = rng.uniform(0.0, 20.0, shape).astype(np.float32)
    r = rng.standard_normal(shape).astype(np.float32)
    out = []
    for blocks in ("16", "8", "2", "1"):
        monkeypatch.setenv("HCA_MG_CLUSTER", blocks)
        sim, cfg, _ = make_pair(shape, "f32", seed=2, n_drugs=1, preconditioner=hca.HCA_PC_MG, picard_maxit=1)
        sim.set_states(st)
        sim.set_field(hca.FIELD_O2, K)
        perf = sim.field(hca.FIELD_PERF).astype(np.float64)
        out.append([sim.apply_preconditioner(w, r) for w in (0, 1)])
        sim.close()
    for which in (0, 1):
        c, a = _system(which, st, K.astype(np.float64), perf, cfg)
        ref = MG.vcycle(MG.hierarchy(c, a), r.astype(np.float64))
        tol = 8 * 2.0 ** -24 * (6 * c + a.max()) / a.mean()
        assert np.max(np.abs(out[0][which] - ref)) <= tol * np.max(np.abs(ref))
        for other in out[1:]:
            assert np.array_equal(out[0][which], other[which])
